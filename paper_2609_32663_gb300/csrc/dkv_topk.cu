// Exact-budget pattern export (Eq. 3, App. A.3): M = TopKMask(P, K), the K
// largest of the n entries of P set to 1. Ties go to the lower flat index and
// NaN ranks below every number (+0 and -0 tie).
//
// Up to kClEntries entries go to the one-cluster kernel further down. More: one
// cooperative launch, a radix select over an order-preserving 32-bit key of
// each value, in phases separated by grid barriers. CTA c owns the contiguous
// index range [lo_c, hi_c) (its warps equal parts of it) and reads it in
// phases 1, 2, 3 and 5 (from L2 after the first, while P fits there).
//   1  histogram of key bits 31-21 (2048 bins);
//   2  every CTA scans that histogram from the top for the bin holding rank K
//      (digit d1, rank k1 left inside it), then histograms bits 20-10 of the
//      keys whose top bits are d1;
//   3  likewise d2, k2, and a histogram of bits 9-0 of the keys matching d1 d2,
//      one per warp range;
//   4  d3 completes the threshold key T; k3 = ties at T to take; the keys equal
//      to T per warp range are bin d3 of that warp's histogram, and each CTA
//      publishes its total;
//   5  M[i] = key > T, or key == T and i is among the first k3 such indices
//      (prefix of the CTA counts, then block scans in index order).
// Histograms build in shared memory; a thread counts runs of equal bins in a
// register and adds a run when its bin changes (patterns are smooth, so runs
// are long), and a CTA adds its nonzero bins to the global histogram.
#include "dkv.h"
#include "dkv_internal.cuh"
#include "dkv_ptx.cuh"

#include <cooperative_groups.h>

#include <cstdint>
#include <mutex>

namespace dkv {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kTkThreads = 512;
constexpr int kTkWarps = kTkThreads / 32;
constexpr int kTkMaxCtas = 2048;
constexpr int kTkMinPerCta = 2048;        // entries per CTA before the grid grows
constexpr int kTkSpins = 1 << 24;         // bound on barrier polls (each an L2 round trip), and 2 s
constexpr int kTkSmem = kTkWarps * 1024 * 4;  // per-warp histograms of the last digit

// Workspace (uint32): status, barrier counter, histograms of the three digit
// passes, per-CTA tie counts.
constexpr int kWsStatus = 0;
constexpr int kWsBarrier = 1;
constexpr int kWsH1 = 16;
constexpr int kWsH2 = kWsH1 + 2048;
constexpr int kWsH3 = kWsH2 + 2048;
constexpr int kWsTies = kWsH3 + 1024;
constexpr int kWsZeroed = kWsTies;  // words cleared before each launch
constexpr int kWsWords = kWsTies + kTkMaxCtas;

__device__ __forceinline__ uint32_t order_key(float x)
{
    if (x != x) return 0u;  // NaN: below every number
    uint32_t u = __float_as_uint(x);
    if (u == 0x80000000u) u = 0u;  // -0 ranks as +0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Grid barrier number `phase` (1, 2, ...): every CTA arrives once per phase on
// a counter zeroed before the launch. Bounded: false after kTkSpins polls (the
// status word is then set), and the caller returns.
__device__ bool grid_barrier(uint32_t* ws, uint32_t phase, uint32_t expected, int* ok_sh)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t* ctr = ws + kWsBarrier;
        __threadfence();  // this CTA's histogram and count writes, ordered by the CTA barrier above
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
        const uint32_t target = phase * expected;
        int ok = 0;
        unsigned long long t0;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
        for (int i = 0; i < kTkSpins; ++i) {
            if (ld_acquire(ctr) >= target) {
                ok = 1;
                break;
            }
            if ((i & 255) == 255) {  // and at most 2 s
                unsigned long long t;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if (t - t0 > 2000000000ull) break;
            }
        }
        if (!ok) atomicOr(ws + kWsStatus, 1u);
        __threadfence();
        *ok_sh = ok;
    }
    __syncthreads();
    return *ok_sh != 0;
}

// Adds the run (bin, cnt) of this thread to the shared histogram.
__device__ __forceinline__ void flush_run(uint32_t* h, uint32_t bin, uint32_t cnt)
{
    if (cnt) atomicAdd(h + bin, cnt);
}

// Keys of the warp's range [wlo, whi) in steps of 32 consecutive entries, eight
// steps' loads issued together (P is read from L2 after the first phase, and
// one load per lane in flight would leave the loop latency bound). f(i, key)
// sees every entry of the range once, in index order within a lane.
template <class F>
__device__ __forceinline__ void for_keys(const float* P, int64_t wlo, int64_t whi, int lane, F f)
{
    constexpr int U = 8;
    for (int64_t i0 = wlo; i0 < whi; i0 += 32 * U) {
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + 32 * u + lane;
            v[u] = i < whi ? __ldg(P + i) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + 32 * u + lane;
            f(i, i < whi, order_key(v[u]));
        }
    }
}

// Histogram of digit (key >> shift) & mask over the warp ranges' keys whose
// bits above the digit equal `prefix` (all keys when pbits == 0), added to the
// global histogram g. PER_WARP: each warp counts into its own hw[warp][nbins]
// (kept for the caller) and the CTA sums them; else one shared h[nbins].
template <bool PER_WARP>
__device__ void histogram(const float* P, int64_t wlo, int64_t whi, int lane, uint32_t* h, int nbins, int shift,
                          uint32_t mask, int pbits, uint32_t prefix, uint32_t* g)
{
    const int nh = PER_WARP ? kTkWarps * nbins : nbins;
    for (int i = threadIdx.x; i < nh; i += blockDim.x) h[i] = 0;
    __syncthreads();
    uint32_t* mine = PER_WARP ? h + (threadIdx.x >> 5) * nbins : h;
    uint32_t run_bin = 0, run_cnt = 0;
    const int pshift = 32 - pbits;
    for_keys(P, wlo, whi, lane, [&](int64_t, bool in, uint32_t key) {
        if (!in || (pbits && (key >> pshift) != prefix)) return;
        const uint32_t bin = (key >> shift) & mask;
        if (bin != run_bin) {
            flush_run(mine, run_bin, run_cnt);
            run_bin = bin;
            run_cnt = 0;
        }
        ++run_cnt;
    });
    flush_run(mine, run_bin, run_cnt);
    __syncthreads();
    for (int i = threadIdx.x; i < nbins; i += blockDim.x) {
        uint32_t c = h[i];
        if (PER_WARP)
            for (int w = 1; w < kTkWarps; ++w) c += h[w * nbins + i];
        if (c) atomicAdd(g + i, c);
    }
}

// The bin of the global histogram g[nbins] that holds rank `rank` (1-based,
// counted from the largest bin down), and the rank left inside it. Every CTA
// computes it from the same counts. Thread t owns bins nbins-1-q t .. nbins-q-q t
// (q = nbins / blockDim, descending).
__device__ void select_bin(const uint32_t* g, int nbins, uint32_t rank, uint32_t* scratch, uint32_t* bin_out,
                           uint32_t* rank_out)
{
    const int q = nbins / kTkThreads;  // 4 or 2
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t c[4], sum = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        c[i] = i < q ? __ldcg(g + nbins - 1 - q * t - i) : 0u;
        sum += c[i];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) scratch[warp] = incl;
    __syncthreads();
    uint32_t before = 0;
    for (int w = 0; w < warp; ++w) before += scratch[w];
    const uint32_t excl = before + incl - sum;
    if (excl < rank && excl + sum >= rank) {  // exactly one thread: the rank lies in its bins
        uint32_t cum = excl;
        for (int i = 0; i < q; ++i) {
            if (cum + c[i] >= rank) {
                *bin_out = (uint32_t)(nbins - 1 - q * t - i);
                *rank_out = rank - cum;
                break;
            }
            cum += c[i];
        }
    }
    __syncthreads();
}

// arrivals: the CTAs each grid barrier counts, gridDim.x (one more only under
// fault injection, so that the first barrier's wait runs out).
__global__ void __launch_bounds__(kTkThreads) topk_kernel(const float* __restrict__ P, int n, uint32_t K,
                                                          uint8_t* __restrict__ M, uint32_t* ws, uint32_t arrivals)
{
    extern __shared__ uint32_t h[];  // [kTkWarps][1024]: phase 3's per-warp histograms; [2048] before
    __shared__ uint32_t scratch[kTkWarps];
    __shared__ uint32_t wties[kTkWarps];
    __shared__ uint32_t sel_bin, sel_rank, base_sh;
    __shared__ int ok_sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // CTA c owns [lo, hi); warp w of it owns the w-th of kTkWarps equal parts.
    const int64_t per = ((int64_t)n + gridDim.x - 1) / gridDim.x;
    const int64_t lo = min((int64_t)n, per * blockIdx.x), hi = min((int64_t)n, lo + per);
    const int64_t wlo = lo + (hi - lo) * warp / kTkWarps, whi = lo + (hi - lo) * (warp + 1) / kTkWarps;

    // 1: top 11 bits
    histogram<false>(P, wlo, whi, lane, h, 2048, 21, 2047u, 0, 0u, ws + kWsH1);
    if (!grid_barrier(ws, 1, arrivals, &ok_sh)) return;
    select_bin(ws + kWsH1, 2048, K, scratch, &sel_bin, &sel_rank);
    const uint32_t d1 = sel_bin, k1 = sel_rank;
    // 2: bits 20-10 of the keys in bin d1
    histogram<false>(P, wlo, whi, lane, h, 2048, 10, 2047u, 11, d1, ws + kWsH2);
    if (!grid_barrier(ws, 2, arrivals, &ok_sh)) return;
    select_bin(ws + kWsH2, 2048, k1, scratch, &sel_bin, &sel_rank);
    const uint32_t p22 = (d1 << 11) | sel_bin, k2 = sel_rank;
    // 3: bits 9-0 of the keys matching the 22-bit prefix, per warp
    histogram<true>(P, wlo, whi, lane, h, 1024, 0, 1023u, 22, p22, ws + kWsH3);
    if (!grid_barrier(ws, 3, arrivals, &ok_sh)) return;
    select_bin(ws + kWsH3, 1024, k2, scratch, &sel_bin, &sel_rank);
    const uint32_t T = (p22 << 10) | sel_bin, take = sel_rank;  // take the first `take` keys equal to T
    // 4: keys equal to T per warp range (bin d3 of the warp's histogram) and per CTA
    if (lane == 0) wties[warp] = h[warp * 1024 + sel_bin];
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (int w = 0; w < kTkWarps; ++w) s += wties[w];
        ws[kWsTies + blockIdx.x] = s;
    }
    if (!grid_barrier(ws, 4, arrivals, &ok_sh)) return;
    // 5: mark. Ties before this warp's range: the earlier CTAs', then the
    // earlier warps' of this CTA; within the range, ballots in index order.
    if (warp == 0) {
        uint32_t b = 0;
        for (int c = lane; c < (int)blockIdx.x; c += 32) b += __ldcg(ws + kWsTies + c);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) b += __shfl_xor_sync(kFull, b, o);
        if (lane == 0) base_sh = b;
    }
    __syncthreads();
    uint32_t carry = base_sh;
    for (int w = 0; w < warp; ++w) carry += wties[w];
    const unsigned below = (1u << lane) - 1u;
    for_keys(P, wlo, whi, lane, [&](int64_t i, bool in, uint32_t key) {
        const bool tie = in && key == T;
        const unsigned bal = __ballot_sync(kFull, tie);
        if (in) M[i] = (key > T || (tie && carry + __popc(bal & below) < take)) ? 1 : 0;
        carry += __popc(bal);
    });
}

// ------------------------------------------------------------ one cluster
// The same select for patterns that one cluster of 8 CTAs holds in registers (KPT
// keys a thread). What bounds the kernel above on those is the latency of its
// phases: a memset launch, a cooperative launch, and four barriers through L2 with P
// and the histograms read through L2 between them. Here P is read once, a phase ends
// in the hardware's cluster barrier, and a digit's histogram of all keys lives in the
// CTAs' shared memory: bin b in CTA b % 8, so that the few bins of a narrow range of
// values spread over the CTAs. (Every CTA reading all eight histograms and adding them
// up, without remote atomics, was slower: 16.2 us at 131,072 entries.)
//
// A CTA counts in kCopies copies of its histogram, lane by lane: the first digit is
// the sign, the exponent and two bits, a dozen bins for probabilities, and without
// copies a warp's lanes would queue for them. Copy c is rotated by 8 c words, so that
// a bin's copies lie in different banks.
//
// A unit of 128 entries is a warp's step, 4 consecutive ones a lane: 16-byte loads and
// 4-byte stores where P and M are aligned for them. The launch overlaps its start with
// the end of the previous kernel.
//
// us a call, grid-wide kernel and this one, probabilities: 1,536 entries 18.9 -> 7.6,
// 65,536 22.6 -> 8.8, 131,072 22.6 -> 11.6, 262,144 23.9 -> 18.6; any bit pattern as
// probabilities within 6 %. (Clusters of 16 CTAs x 512 threads: 11.6 at 131,072 but 14.9
// for uniform bit patterns, whose 2,048 bins are all remote additions; 8 x 512 12.8, 4 x
// 1,024 17.3.)
constexpr int kClCtas = 8, kClThreads = 1024, kClWarps = kClThreads / 32;
constexpr int kClBins = 2048, kCopies = 4, kClUnit = 128;
constexpr int kClSmem = kCopies * kClBins * 4;
constexpr int kClOwn = kClBins / kClCtas;

template <int KPT>
__global__ void __launch_bounds__(kClThreads, 1) topk_cluster_kernel(const float* __restrict__ P, int n, uint32_t K,
                                                                     uint8_t* __restrict__ M, uint32_t* ws)
{
    namespace cg = cooperative_groups;
    constexpr int U = KPT / 4;                        // units a warp
    extern __shared__ __align__(16) uint32_t hist[];  // [kCopies][kClBins]
    __shared__ uint32_t tot[3][kClOwn];               // of each digit: this CTA's bins of the whole histogram
    __shared__ uint32_t warp_sum[kClWarps], wties[kClWarps], cta_ties[kClCtas];
    __shared__ uint32_t sel_bin, sel_rank;
    const cg::cluster_group cluster = cg::this_cluster();
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int rank = (int)cluster.block_rank();
    // The units of CTA `rank`, and of them those of this warp: at most U.
    const int units = (n + kClUnit - 1) / kClUnit;
    const int u0 = units * rank / kClCtas, u1 = units * (rank + 1) / kClCtas;
    const int wlo = kClUnit * (u0 + (u1 - u0) * warp / kClWarps) + 4 * lane;  // the lane's first entry
    const int whi = min(n, kClUnit * (u0 + (u1 - u0) * (warp + 1) / kClWarps));
    const bool vec_p = (reinterpret_cast<uintptr_t>(P) & 15u) == 0, vec_m = (reinterpret_cast<uintptr_t>(M) & 3u) == 0;

    for (int i = t; i < kClBins * kCopies / 4; i += kClThreads) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = t; i < 3 * kClOwn; i += kClThreads) (&tot[0][0])[i] = 0u;
    cluster.barrier_arrive();
    // Overlaps its start with the previous kernel's end; that kernel's results are read from here on.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (rank == 0 && t == 0) ws[kWsStatus] = 0u;
    float4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int i = wlo + kClUnit * u;
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (vec_p && i + 3 < whi) {
            v[u] = ld_prev(reinterpret_cast<const float4*>(P + i));
        } else {
            if (i < whi) v[u].x = ld_prev(P + i);
            if (i + 1 < whi) v[u].y = ld_prev(P + i + 1);
            if (i + 2 < whi) v[u].z = ld_prev(P + i + 2);
            if (i + 3 < whi) v[u].w = ld_prev(P + i + 3);
        }
    }
    uint32_t key[KPT];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        key[4 * u] = order_key(v[u].x);
        key[4 * u + 1] = order_key(v[u].y);
        key[4 * u + 2] = order_key(v[u].z);
        key[4 * u + 3] = order_key(v[u].w);
    }
    const auto valid = [&](int i) { return wlo + kClUnit * (i >> 2) + (i & 3) < whi; };
    cluster.barrier_wait();  // every CTA's bins are zero

    // Digit by digit from the top: bits 31-21, 20-10, 9-0.
    uint32_t prefix = 0, k = K;  // the bits of the K-th key known so far, and its rank among the keys that have them
    const int copy = lane & (kCopies - 1);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        constexpr int kShift[3] = {21, 10, 0};
        const int bits = d < 2 ? 11 : 10, shift = kShift[d], nbins = 1 << bits;
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            if (valid(i) && (d == 0 || (key[i] >> (shift + bits)) == prefix)) {
                const uint32_t bin = (key[i] >> shift) & (uint32_t)(nbins - 1);
                atomicAdd(hist + copy * kClBins + ((bin + 8 * copy) & (kClBins - 1)), 1u);
            }
        __syncthreads();
#pragma unroll
        for (int b = t; b < nbins; b += kClThreads) {
            uint32_t c = 0;
#pragma unroll
            for (int r = 0; r < kCopies; ++r) {
                uint32_t* h = hist + r * kClBins + ((b + 8 * r) & (kClBins - 1));
                c += *h;
                *h = 0u;  // for the next digit
            }
            if (c) atomicAdd(cluster.map_shared_rank(&tot[d][b / kClCtas], b % kClCtas), c);
        }
        cluster.sync();
        // The bin that holds rank k, counted from the largest down, and the rank inside
        // it. Thread t has the q bins nbins - 1 - q t downwards.
        const int q = nbins / kClThreads;
        uint32_t c[kClBins / kClThreads], sum = 0;
#pragma unroll
        for (int i = 0; i < q; ++i) {
            const int b = nbins - 1 - q * t - i;
            c[i] = *cluster.map_shared_rank(&tot[d][b / kClCtas], b % kClCtas);
            sum += c[i];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        const uint32_t excl = __reduce_add_sync(kFull, lane < warp ? warp_sum[lane & (kClWarps - 1)] : 0u) + incl - sum;
        if (excl < k && excl + sum >= k) {  // exactly one thread
            uint32_t above = excl;
            bool found = false;
#pragma unroll
            for (int i = 0; i < q; ++i) {
                if (!found && above + c[i] >= k) {
                    sel_bin = (uint32_t)(nbins - 1 - q * t - i);
                    sel_rank = k - above;
                    found = true;
                }
                above += c[i];
            }
        }
        __syncthreads();
        prefix = (prefix << bits) | sel_bin;
        k = sel_rank;
    }

    // The threshold key is prefix; the first k keys equal to it are taken, in index order.
    uint32_t ties = 0;  // bit i: key i of this thread is one
#pragma unroll
    for (int i = 0; i < KPT; ++i) ties |= valid(i) && key[i] == prefix ? 1u << i : 0u;
    const uint32_t of_warp = __reduce_add_sync(kFull, (uint32_t)__popc(ties));
    if (lane == 0) wties[warp] = of_warp;
    __syncthreads();
    if (warp == 0) {
        const uint32_t all = __reduce_add_sync(kFull, lane < kClWarps ? wties[lane] : 0u);
        if (lane < kClCtas) *cluster.map_shared_rank(&cta_ties[rank], lane) = all;
    }
    cluster.sync();  // the last access to another CTA's shared memory is before it
    uint32_t carry =
        __reduce_add_sync(kFull, (lane < warp ? wties[lane & (kClWarps - 1)] : 0u) + (lane < rank ? cta_ties[lane & (kClCtas - 1)] : 0u));
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const uint32_t here = (ties >> (4 * u)) & 15u;
        uint32_t take = 0;  // the lane's ties of this unit that are taken
        if (__any_sync(kFull, here != 0)) {
            uint32_t incl = __popc(here);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t x = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += x;
            }
            uint32_t before = carry + incl - __popc(here);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if ((here >> j) & 1u) take |= before++ < k ? 1u << j : 0u;
            carry += __shfl_sync(kFull, incl, 31);
        }
        uchar4 m;
        m.x = key[4 * u] > prefix || (take & 1u);
        m.y = key[4 * u + 1] > prefix || (take & 2u);
        m.z = key[4 * u + 2] > prefix || (take & 4u);
        m.w = key[4 * u + 3] > prefix || (take & 8u);
        const int i = wlo + kClUnit * u;
        if (vec_m && i + 3 < whi) {
            *reinterpret_cast<uchar4*>(M + i) = m;
        } else {
            if (i < whi) M[i] = m.x;
            if (i + 1 < whi) M[i + 1] = m.y;
            if (i + 2 < whi) M[i + 2] = m.z;
            if (i + 3 < whi) M[i + 3] = m.w;
        }
    }
}

// The most entries: 32 keys a thread. Beyond, 16 CTAs would be needed, which is a cluster
// size that a device need not have, for 28.7 -> 25.7 us at 393,216.
constexpr int kClMaxKeys = 32;
constexpr int kClEntries = kClCtas * kClThreads * kClMaxKeys;

using TopkClusterFn = void (*)(const float*, int, uint32_t, uint8_t*, uint32_t*);
TopkClusterFn cluster_kernel(int64_t n)
{
    // The fewest keys a thread that hold n: every one is a step of each loop (131,072
    // entries 11.6 us with 16, 65,536 8.8 with 8).
    return n <= kClCtas * kClThreads * 8    ? topk_cluster_kernel<8>
           : n <= kClCtas * kClThreads * 16 ? topk_cluster_kernel<16>
                                            : topk_cluster_kernel<kClMaxKeys>;
}

void cluster_config(cudaLaunchConfig_t* lc, cudaLaunchAttribute* attr, cudaStream_t st)
{
    *lc = {};
    lc->gridDim = dim3(kClCtas);
    lc->blockDim = dim3(kClThreads);
    lc->dynamicSmemBytes = kClSmem;
    lc->stream = st;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = kClCtas;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    lc->attrs = attr;
    lc->numAttrs = 2;
}

// The kernels' attributes, and whether the device (or this process's share of it)
// can run a cluster of this size.
cudaError_t setup_cluster(bool* usable)
{
    *usable = true;
    for (const int64_t n : {(int64_t)1, (int64_t)kClEntries / 2, (int64_t)kClEntries}) {
        const TopkClusterFn f = cluster_kernel(n);
        cudaError_t e;
        if ((e = cudaFuncSetAttribute((const void*)f, cudaFuncAttributeMaxDynamicSharedMemorySize, kClSmem)) != cudaSuccess)
            return e;
        cudaLaunchConfig_t lc;
        cudaLaunchAttribute attr[2];
        cluster_config(&lc, attr, nullptr);
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, (const void*)f, &lc) != cudaSuccess) {
            cudaGetLastError();
            clusters = 0;
        }
        *usable = *usable && clusters > 0;
    }
    return cudaSuccess;
}

}  // namespace

int64_t topk_workspace_bytes() { return (int64_t)kWsWords * 4; }

cudaError_t launch_topk(const float* P, int64_t n, int64_t K, uint8_t* M, void* workspace, cudaStream_t st,
                        bool phantom_cta)
{
    cudaError_t e;
    if (n == 0) return cudaSuccess;
    if (K == 0 || K == n) return cudaMemsetAsync(M, K == n ? 1 : 0, (size_t)n, st);
    uint32_t* ws = static_cast<uint32_t*>(workspace);
    // Device capacity, looked up once per device (the host cost of these calls
    // would otherwise dominate small exports).
    static std::mutex mu;
    static int cached_dev = -1, cached_cap = 0;
    static bool cached_cluster = false;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    int64_t cap = 0;
    bool cluster = false;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (cached_dev != dev) {
            int sms = 0, per_sm = 0;
            if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
            if ((e = cudaFuncSetAttribute(topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTkSmem)) !=
                cudaSuccess)
                return e;
            if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, topk_kernel, kTkThreads, kTkSmem)) !=
                cudaSuccess)
                return e;
            if ((e = setup_cluster(&cached_cluster)) != cudaSuccess) return e;
            cached_cap = sms * (per_sm < 1 ? 1 : per_sm);
            cached_dev = dev;
        }
        cap = cached_cap;
        cluster = cached_cluster;
    }
    // (The barrier's fault injection is the other kernel's.)
    if (cluster && n <= kClEntries && !phantom_cta) {
        cudaLaunchConfig_t lc;
        cudaLaunchAttribute attr[2];
        cluster_config(&lc, attr, st);
        return cudaLaunchKernelEx(&lc, cluster_kernel(n), P, (int)n, (uint32_t)K, M, ws);
    }
    if ((e = cudaMemsetAsync(ws, 0, sizeof(uint32_t) * kWsZeroed, st)) != cudaSuccess) return e;
    // Every CTA must be resident at once (grid barriers): at most the device's
    // capacity, and no more CTAs than ranges of kTkMinPerCta entries.
    const int64_t want = (n + kTkMinPerCta - 1) / kTkMinPerCta;
    int grid = (int)(want < cap ? want : cap);
    if (grid > kTkMaxCtas) grid = kTkMaxCtas;
    if (grid < 1) grid = 1;
    int nn = (int)n;
    uint32_t KK = (uint32_t)K;
    uint32_t arrivals = (uint32_t)grid + (phantom_cta ? 1u : 0u);
    void* args[] = {(void*)&P, (void*)&nn, (void*)&KK, (void*)&M, (void*)&ws, (void*)&arrivals};
    return cudaLaunchCooperativeKernel((const void*)topk_kernel, dim3(grid), dim3(kTkThreads), args, kTkSmem, st);
}

}  // namespace dkv
