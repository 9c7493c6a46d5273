// Pieces shared by the decode kernels (split-K over the packed cache, Sec. 3.4):
// programmatic-dependent-launch wrappers (the mbarrier and bulk-copy ones are in
// dkv_ptx.cuh), the per-call slab table, the stream-K row partition over the slabs of one layer, the tile cursor of a
// warp, and the end of a CTA's pass: merging the warp states that share a slab
// and the fused cross-CTA merge (the last CTA of a slab merges every CTA's
// partial of it).
#pragma once

#include "dkv_internal.cuh"
#include "dkv_ptx.cuh"

#include <math.h>

namespace dkv {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxB = 512;
constexpr float kSlack = 8.f;        // lazy-rescale threshold of the online softmax (log2 units)

// A value that is the same in every lane, read from lane 0. The compiler then
// knows it is uniform over the warp: loops and branches on it are plain ones (the
// warp-wide votes and shuffles inside need no check for a split warp), and the
// scalar work on it runs once a warp, in uniform registers.
__device__ __forceinline__ int uniform(int x) { return __shfl_sync(kFull, x, 0); }

// Programmatic dependent launch: let the next kernel in the stream start its
// prologue, and wait for the previous kernel's results before reading them.
__device__ __forceinline__ void pdl_launch_dependents()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ void pdl_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ------------------------------------------------------------ partition
// Per-call sequence table in shared memory: NA[b] = rows already appended
// (clamped to the reserve), NP[b] = exclusive prefix over b of the extra rows
// e_b = NA[b] + (this call appends to b ? 1 : 0). Layer rows fit in int32.
//
// When the layer has fewer than kSlabCache slabs, the table also holds the
// slabs' first layer rows P0[h] ([NHl+1], the extra rows included) and cache
// offsets OFF[h] = off[h] ([NHl]), so that finding a warp's rows and streaming
// them reads no plan metadata from global memory: a CTA that starts after the
// previous kernel has drained (the last ones to get an SM) would otherwise pay
// a chain of dependent L2 round trips, under full HBM load, before its first
// copy. P0 and OFF are null for larger layers (computed from global memory then).
constexpr int kSlabCache = 1008;
struct SeqTable {
    int32_t* NA;   // [B]
    int32_t* NP;   // [B+1]
    int32_t* P0;   // [NHl+1] or null
    int64_t* OFF;  // [NHl] or null
};

// Bytes of the table of a layer of B sequences and NHl slabs, at an 8-byte
// aligned base: OFF, P0 (both only when cached), NA, NP.
__host__ __device__ constexpr int seq_table_bytes(int B, int NHl)
{
    return (NHl < kSlabCache ? NHl * 12 + 4 : 0) + (2 * B + 1) * 4;
}
// The most any layer of B sequences needs.
__host__ __device__ constexpr int seq_table_bytes(int B) { return seq_table_bytes(B, kSlabCache - 1); }

__device__ __forceinline__ SeqTable seq_table_at(unsigned char* base, const DecodeArgs& a)
{
    SeqTable t;
    const int NHl = a.B * a.Hkv;
    const bool cached = NHl < kSlabCache;
    t.OFF = cached ? reinterpret_cast<int64_t*>(base) : nullptr;
    t.P0 = cached ? reinterpret_cast<int32_t*>(base + NHl * 8) : nullptr;
    t.NA = reinterpret_cast<int32_t*>(base + (cached ? NHl * 12 + 4 : 0));
    t.NP = t.NA + a.B;
    return t;
}

// Fill P0 (context rows only, so far) and OFF (when cached) with the threads
// [t0, t0 + nt) of the CTA; the caller's barrier publishes them.
__device__ __forceinline__ void load_slab_cache(const DecodeArgs& a, SeqTable t, int t0, int nt)
{
    if (!t.P0) return;
    const int NHl = a.B * a.Hkv;
    const int64_t i0 = __ldg(a.ioff);
#pragma unroll 1
    for (int h = (int)threadIdx.x - t0; h <= NHl; h += nt) {
        t.P0[h] = (int)(__ldg(a.ioff + h) - i0);
        if (h < NHl) t.OFF[h] = __ldg(a.off + h);
    }
}

// Rows that come before slab h in the layer beyond the context rows: NP is ready.
__device__ __forceinline__ int extra_before(const int32_t* NP, int Hkv, int h)
{
    const int b = h / Hkv, g = h - b * Hkv;
    int p = Hkv * NP[b];
    if (g) p += g * (NP[b + 1] - NP[b]);
    return p;
}

// After the barrier that publishes NP and P0's context rows: P0 becomes the
// slabs' first layer rows (all nt threads of the CTA; the caller's next barrier
// publishes it).
__device__ __forceinline__ void finish_slab_cache(const DecodeArgs& a, SeqTable t, int nt)
{
    if (!t.P0) return;
#pragma unroll 1
    for (int h = threadIdx.x; h <= a.B * a.Hkv; h += nt) t.P0[h] += extra_before(t.NP, a.Hkv, h);
}

__device__ void build_seq_table(const DecodeArgs& a, SeqTable t, bool report)
{
    // Called by one full warp.
    const int lane = threadIdx.x & 31;
    int carry = 0;
#pragma unroll 1
    for (int b0 = 0; b0 < a.B; b0 += 32) {
        const int b = b0 + lane;
        int na = 0, e = 0;
        if (b < a.B) {
            const int raw = a.n_app ? a.n_app[b] : 0;
            na = min(max(raw, 0), a.reserve);
            const bool app = a.append && raw >= 0 && raw < a.reserve;
            if (a.append && !app && report) atomicOr(a.status, 0x1 /* DKV_DEV_APPEND_OVERFLOW */);
            e = na + (app ? 1 : 0);
            t.NA[b] = na;
        }
        int incl = e;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        if (b < a.B) t.NP[b] = carry + incl - e;
        carry += __shfl_sync(kFull, incl, 31);
    }
    if (lane == 0) t.NP[a.B] = carry;
}

// First layer row of slab h (h in [0, B*Hkv]) within this call.
// (Out of line: its code would otherwise be repeated at every use.)
__device__ __noinline__ int slab_start_global(const int64_t* ioff, const int32_t* NP, int Hkv, int h)
{
    return (int)(ioff[h] - ioff[0]) + extra_before(NP, Hkv, h);
}

__device__ __forceinline__ int slab_start(const DecodeArgs& a, const SeqTable& t, int h)
{
    return t.P0 ? t.P0[h] : slab_start_global(a.ioff, t.NP, a.Hkv, h);
}

// CTAs that get rows when R > 0 rows are cut into at most P ranges: the first
// live_parts of the grid, each with at least one row.
__device__ __forceinline__ int live_parts(int R, int P) { return min(P, max(R, 1)); }

__device__ __forceinline__ int part_start(int w, int R, int P)
{
    // floor(w R / P) without a 64-bit division: R = q P + r, so w R / P = w q + w r / P,
    // and w r < P^2 fits 32 bits (P is a CTA count).
    const unsigned q = (unsigned)R / (unsigned)P, r = (unsigned)R - q * (unsigned)P;
    return (int)((unsigned)w * q + ((unsigned)w * r) / (unsigned)P);
}

// Largest part w with part_start(w) <= x, for 0 <= x < R. part_start(w) <= x
// exactly when w R < (x + 1) P, so w = floor(((x + 1) P - 1) / R): a float
// estimate of that quotient, then exact integer steps (a chain of integer
// divisions here would put ~0.5 us on the end of every launch).
__device__ __forceinline__ int part_of(int x, int R, int P)
{
    const int64_t num = (int64_t)(x + 1) * P - 1;
    int w = (int)((float)num * __fdividef(1.f, (float)R));
#pragma unroll 1
    while ((int64_t)(w + 1) * R <= num) ++w;
#pragma unroll 1
    while (w > 0 && (int64_t)w * R > num) --w;
    return min(w, P - 1);
}

// Last slab h in [0, NHl) with slab_start(h) <= x.
__device__ int slab_containing(const DecodeArgs& a, const SeqTable& t, int NHl, int x)
{
    int lo = 0, hi = NHl - 1;
#pragma unroll 1
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (slab_start(a, t, mid) <= x)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// ------------------------------------------------------------ softmax helpers
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Tile cursor of one warp over its row range, with the current slab's constants
// (warp-uniform; advanced by the whole warp).
struct Cursor {
    int h;         // slab; == hend when exhausted
    int s0, s1;    // the warp's rows of this slab, [s0, s1) (layer rows)
    int p0;        // slab_start(h)
    int x;         // first row of the current tile
    int n_h;       // rows of the slab in this call
    int app;       // this call appends the slab's last row from k_new/v_new
    int64_t base;  // off[h]: cache row of the slab's first row
};

__device__ __forceinline__ void cursor_seek(Cursor& cu, const DecodeArgs& a, const SeqTable& t, int hend, int wA,
                                            int wB)
{
#pragma unroll 1
    while (cu.h < hend) {
        cu.p0 = uniform(slab_start(a, t, cu.h));
        const int p1 = uniform(slab_start(a, t, cu.h + 1));
        cu.s0 = max(wA, cu.p0);
        cu.s1 = min(wB, p1);
        if (cu.s0 < cu.s1) {
            const int b = cu.h / a.Hkv;
            const int e = t.NP[b + 1] - t.NP[b];
            const int64_t base = t.OFF ? t.OFF[cu.h] : a.off[cu.h];
            cu.n_h = p1 - cu.p0;
            cu.app = uniform((a.append && e > t.NA[b]) ? 1 : 0);
            cu.base = (int64_t)(((uint64_t)(uint32_t)uniform((int)(base >> 32)) << 32) | (uint32_t)uniform((int)base));
            cu.x = cu.s0;
            return;
        }
        ++cu.h;
    }
}

template <int TR>
__device__ __forceinline__ void cursor_next(Cursor& cu, const DecodeArgs& a, const SeqTable& t, int hend, int wA,
                                            int wB)
{
    cu.x += TR;
    if (cu.x < cu.s1) return;
    ++cu.h;
    cursor_seek(cu, a, t, hend, wA, wB);
}

// ------------------------------------------------------------ segments
// A warp's rows of one slab.
struct Segment {
    int h;      // slab
    int left;   // rows (of the segment) from `row` on
    int row;    // cache row of the first of them
    int p0, p1; // the slab's layer rows
    int app;    // the segment's last row is this step's new token
    int settled; // of the segment's rows, from the first, those that the wait need not precede
};

// How many of the layer rows [s0, s1) of a slab that ends at p1, from s0 on, may be
// fetched before the wait for the previous kernel: all of them if no earlier call
// appended to the slab (na rows), else those of the context (all but the extra rows at
// its end). An earlier decode call lets the next kernel start before its appended row
// is stored, so such rows are fetched only after the wait. (This call's own new row
// comes from k_new and v_new.)
__device__ __forceinline__ int settled_rows(int na, int extra, int s0, int s1, int p1)
{
    return na > 0 ? max(0, min(s1, p1 - extra) - s0) : s1 - s0;
}

constexpr int kSegmentWords = 8;  // of a warp's segment slot (7 used)

// The first segment of a slab in [h, hend), which has one, of a warp with the
// layer rows [wA, wB), into the warp's slot in shared memory. (Returned that way,
// not through a local variable: a stack frame of the decode kernels is more than
// the L1 that their shared memory leaves, and a reload from L2 under full load
// costs up to 1 us.)
__device__ __noinline__ void find_segment(const DecodeArgs& a, unsigned char* table, int h, int hend, int wA, int wB,
                                          int32_t* slot)
{
    const SeqTable t = seq_table_at(table, a);
    int p0 = slab_start(a, t, h), p1 = p0;
#pragma unroll 1
    for (; h < hend; ++h, p0 = p1) {
        p1 = slab_start(a, t, h + 1);
        if (max(wA, p0) < min(wB, p1)) break;
    }
    const int s0 = max(wA, p0), s1 = min(wB, p1), b = h / a.Hkv;
    const int na = t.NA[b], extra = t.NP[b + 1] - t.NP[b];
    const int64_t off = t.OFF ? t.OFF[h] : a.off[h];
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        slot[0] = h;
        slot[1] = s1 - s0;
        slot[2] = (int)(off + (s0 - p0));
        slot[3] = p0;
        slot[4] = p1;
        slot[5] = (a.append && s1 == p1 && extra > na) ? 1 : 0;
        slot[6] = settled_rows(na, extra, s0, s1, p1);
    }
    __syncwarp();
}

__device__ __forceinline__ Segment read_segment(const int32_t* slot)
{
    return {uniform(slot[0]), uniform(slot[1]), uniform(slot[2]), uniform(slot[3]), uniform(slot[4]), uniform(slot[5]),
            uniform(slot[6])};
}

// Slabs of the warp's first and last row.
__device__ __noinline__ int2 slab_range(const DecodeArgs& a, unsigned char* table, int wA, int wB)
{
    const SeqTable t = seq_table_at(table, a);
    const int NHl = a.B * a.Hkv;
    return make_int2(slab_containing(a, t, NHl, wA), slab_containing(a, t, NHl, wB - 1));
}

// Number of CTAs whose row range overlaps [p0, p1) (p0 < p1), and the first and
// last of them (R >= P: every CTA has rows).
__device__ __forceinline__ int ctas_of_slab(int p0, int p1, int R, int P, int* c0_out, int* c1_out)
{
    const int c0 = part_of(p0, R, P), c1 = part_of(p1 - 1, R, P);
    *c0_out = c0;
    *c1_out = c1;
    return c1 - c0 + 1;
}

// Output row of column c of slab (b, g): query c / G, head g G + c % G of out [B][Q][H][128].
template <int G>
__device__ __forceinline__ int64_t out_row(const DecodeArgs& a, int b, int g, int c)
{
    const int qi = c / G, j = c - qi * G;
    return ((int64_t)b * a.Q + qi) * a.H + g * G + j;
}

// out row of column c = O / L; O, L of the column for the lane's 4 dims.
template <int G>
__device__ __forceinline__ void write_out(const DecodeArgs& a, int b, int g, int c, float4 O, float L, int lane)
{
    const float inv = L > 0.f ? 1.f / L : 0.f;
    float4* dst = reinterpret_cast<float4*>(a.out + out_row<G>(a, b, g, c) * kHeadDim);
    dst[lane] = make_float4(O.x * inv, O.y * inv, O.z * inv, O.w * inv);
}

// ------------------------------------------------------------ cross-CTA merge
// A slab whose rows lie in several CTAs is merged by the last of them (by index):
// every other CTA leaves its partial (m, l, o) of a column in its slot of the
// fused-merge exchange (a CTA leaves one slab's at most: that of its last slab, if rows
// of it follow in the next CTA), and the merging CTA polls the slots until every word
// has arrived. A slot's words carry their own arrival: an empty word is 0, and a
// partial's zeros are written as -0, so a word is data as soon as it differs from
// 0, whatever order the stores arrive in. That takes one store and one load
// through L2, where an arrival counter took a fence, an atomic, an acquire and
// then the loads: at 32K (50 MB layers) 9.3 us of streaming was followed by up
// to 5.1 us of merge, now 3.3. The merging CTA empties the slots again for the
// next launch (ordered by the launches' dependency). It waits only for CTAs of
// lower index. Where the device holds the whole grid (one CTA an SM) they all run at
// once; elsewhere this assumes that CTAs start in the order of their index, as they do
// but as CUDA does not promise. If that fails the wait runs out: the outputs stay
// unwritten and the status word says so. A partial that arrives after its merge gave up
// stays in the exchange until the status word is cleared (dkv_plan_status empties the
// exchange then): until that, no output of the plan is to be trusted.
__device__ __forceinline__ float full_word(float x) { return __float_as_uint(x) == 0u ? -0.f : x; }

__device__ __forceinline__ bool is_full(const float4& v)
{
    return __float_as_uint(v.x) != 0u && __float_as_uint(v.y) != 0u && __float_as_uint(v.z) != 0u &&
           __float_as_uint(v.w) != 0u;
}

__device__ __forceinline__ float4 ld_exchange4(const float* p)
{
    float4 v;
    asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

__device__ __forceinline__ float2 ld_exchange2(const float* p)
{
    float2 v;
    asm volatile("ld.relaxed.gpu.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_exchange4(float* p, float4 v)
{
    asm volatile("st.relaxed.gpu.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

__device__ __forceinline__ void st_exchange2(float* p, float x, float y)
{
    asm volatile("st.relaxed.gpu.global.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(x), "f"(y) : "memory");
}

// Bound of a poll loop over the exchange, decided by the whole warp: true once the
// polls or the time since the 64th poll run out.
__device__ __forceinline__ bool polled_out(int spin, unsigned long long& t0)
{
    if ((spin & 63) != 0) return false;
    const unsigned long long now = global_ns();
    if (t0 == 0) t0 = now;
    return __any_sync(kFull, spin >= kWaitSpins || now - t0 > kWaitNs);
}

// One warp writes CTA c's partial of column j.
__device__ __forceinline__ void put_partial(const DecodeArgs& a, int c, int j, int NC, float4 O, float M, float L, int lane)
{
    const int64_t sj = (int64_t)c * NC + j;
    st_exchange4(a.exch_o + sj * kHeadDim + 4 * lane,
                 make_float4(full_word(O.x), full_word(O.y), full_word(O.z), full_word(O.w)));
    if (lane == 0) st_exchange2(a.exch_ml + sj * 2, full_word(M), full_word(L));
}

// One warp of the merging CTA adds to a state (M, L, O: 4 dims a lane) of column
// j of a slab the partials of the CTAs first, first + step, ... below end (step 1
// or 2), KB at a time, and empties their slots. A batch is one round trip to L2
// (0.5 us) once its words are there: lane k reads the k-th partial's m and l,
// every lane its dims of all of them. KB = 12: with 8 a slab of 19 CTAs takes a
// second round (128K 1,026 -> 1,040 us per step, 4K 261 -> 280), 16 is no faster.
// False when a partial did not arrive within the wait bound.
template <int KB, int NCC>
__device__ __forceinline__ bool merge_partials(const DecodeArgs& a, int j, int NC_, int first, int step,
                                               int end, float& M, float& L, float4& O, int lane)
{
    const int NC = NCC ? NCC : NC_;
    const int stride = step * NC;
    const int64_t base = (int64_t)first * NC + j;
    float* po = a.exch_o + base * kHeadDim + 4 * lane;
    float* pm = a.exch_ml + (base + (int64_t)lane * stride) * 2;
    bool good = true;
    float Lk = 0.f;  // this lane's share of the partials' sums
#pragma unroll 1
    for (int n = (end - first + step - 1) >> (step - 1); n > 0;
         n -= KB, po += KB * stride * kHeadDim, pm += KB * stride * 2) {
        float4 v[KB];
        float2 ml;
        unsigned long long t0 = 0;
#pragma unroll 1
        for (int spin = 1;; ++spin) {
            ml = make_float2(-INFINITY, -0.f);
            if (lane < min(n, KB)) ml = ld_exchange2(pm);
            // Slots past the last one read the first again: no branches.
#pragma unroll
            for (int u = 0; u < KB; ++u) v[u] = ld_exchange4(po + (u < n ? u * stride * kHeadDim : 0));
            bool full = __float_as_uint(ml.x) != 0u && __float_as_uint(ml.y) != 0u;
#pragma unroll
            for (int u = 0; u < KB; ++u) full &= is_full(v[u]);
            if (__all_sync(kFull, full)) break;
            if (polled_out(spin, t0)) {
                good = false;
                break;
            }
        }
        float Mb = fmaxf(M, ml.x);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) Mb = fmaxf(Mb, __shfl_xor_sync(kFull, Mb, o));
        const float fo = (M == -INFINITY) ? 0.f : ex2(M - Mb);
        const float f = (ml.x == -INFINITY) ? 0.f : ex2(ml.x - Mb);
        M = Mb;
        L *= fo;
        Lk = fmaf(Lk, fo, f * ml.y);
        O.x *= fo;
        O.y *= fo;
        O.z *= fo;
        O.w *= fo;
#pragma unroll
        for (int u = 0; u < KB; ++u) {
            const float fu = __shfl_sync(kFull, f, u);
            if (u < n) {
                O.x = fmaf(fu, v[u].x, O.x);
                O.y = fmaf(fu, v[u].y, O.y);
                O.z = fmaf(fu, v[u].z, O.z);
                O.w = fmaf(fu, v[u].w, O.w);
                st_exchange4(po + u * stride * kHeadDim, make_float4(0.f, 0.f, 0.f, 0.f));
            }
        }
        if (lane < min(n, KB)) st_exchange2(pm, 0.f, 0.f);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) Lk += __shfl_xor_sync(kFull, Lk, o);
    L += Lk;
    if (!good && lane == 0) atomicOr(a.status, 0x4 /* DKV_DEV_MERGE_TIMEOUT */);
    return good;
}

// End of a CTA's pass after a copy that never landed: its outputs stay unwritten
// (the status word says so), but the slabs it shares with other CTAs still get
// their exchange words, as an empty partial, or are collected, so that no other
// CTA waits for this one and the next launch finds the exchange empty.
template <int NW>
__device__ __noinline__ void dead_tail(const DecodeArgs& a, const SeqTable& tab, int NC, int c, int A, int Bc, int R,
                                       int P, int warp, int lane)
{
    const int NHl = a.B * a.Hkv;
    const int hf = slab_containing(a, tab, NHl, A), hl = slab_containing(a, tab, NHl, Bc - 1);
#pragma unroll 1
    for (int e = 1; e >= 0; --e) {  // the last slab first: its partial waits for nobody
        const int h = e ? hl : hf;
        if (e && hl == hf) continue;
        int c0, c1;
        if (ctas_of_slab(slab_start(a, tab, h), slab_start(a, tab, h + 1), R, P, &c0, &c1) <= 1) continue;
#pragma unroll 1
        for (int j = warp; j < NC; j += NW) {
            float M = -INFINITY, L = 0.f;
            float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
            if (c1 == c)
                merge_partials<4, 0>(a, j, NC, c0, 1, c1, M, L, O, lane);
            else
                put_partial(a, c, j, NC, O, M, L, lane);
        }
    }
}

__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// What a CTA records for its end (int32 words in shared memory): seg_first[NW],
// seg_last[NW] (first / last slab of warp w, -1 if none), the layer rows [p0, p1)
// of each entry (2 w: first, 2 w + 1: last) as p0[2 NW], p1[2 NW], whether a warp
// gave up a copy wait, and the first CTA of the CTA's first slab.
template <int NW>
struct TailMeta {
    static constexpr int kFirst = 0, kLast = NW, kP0 = 2 * NW, kP1 = 4 * NW, kDead = 6 * NW, kC0 = 6 * NW + 1;
    static constexpr int kWords = 6 * NW + 4;
};

// End of one CTA's split-K pass over the layer rows [A, Bc), after its warps'
// ranges are done and a CTA barrier. NCC: the number of columns per slab when
// fixed at compile time (the decode step: G), 0 to take a.NC. The first slab's
// state of warp w is in the warp record (c, w) of warp_o / warp_ml, the last
// slab's in its own ring at ring + w * ring_bytes (o[NC][128] then (m, l)[NC]);
// the ring has 528 free bytes at dep_off. The states of each slab are merged; a
// slab wholly inside this CTA is written out (fused). Otherwise the CTA leaves its partial in the exchange,
// or, as the slab's last CTA, merges everyone's; not fused, the CTA writes its
// partial to slot c + h of the workspace.
//
// A task is (slab, column), one warp each: it merges the CTA's own states. While
// there are at least twice (three times) as many warps as tasks, a task has one
// (two) more warps, which meanwhile collect the other CTAs' partials. With fewer
// warps the tasks run from the CTA's last slab to its first, the only one it can
// be the last CTA of: what others wait for is written before this CTA waits.
template <int G, int NW, bool FUSED, int NCC>
__device__ __forceinline__ void cta_tail(const DecodeArgs& a, unsigned char* ring, int ring_bytes, int dep_off,
                                         const int32_t* meta, int c, int A, int Bc, int warp, int lane)
{
    using TM = TailMeta<NW>;
    // Entry e (lane e) is the first (even e) or last (odd e) slab of warp e/2, -1 if
    // none; entries list their slabs in non-decreasing order.
    static_assert(2 * NW <= 32, "one entry per lane");
    int h_e = -1, p0_e = 0, p1_e = 0;
    if (lane < 2 * NW) {
        h_e = meta[((lane & 1) ? TM::kLast : TM::kFirst) + (lane >> 1)];
        p0_e = meta[TM::kP0 + lane];
        p1_e = meta[TM::kP1 + lane];
    }
    // Slab of the nearest valid entry before this one (-1 if none): one ballot
    // and one shuffle.
    const unsigned valid = __ballot_sync(kFull, h_e >= 0);
    const unsigned below = valid & ((1u << lane) - 1u);
    const int hprev = __shfl_sync(kFull, h_e, below ? 31 - __clz(below) : 0);
    const int prev = below ? hprev : -1;
    const unsigned fresh = __ballot_sync(kFull, h_e >= 0 && h_e != prev);
    const int nslab = uniform(__popc(fresh));
    const int NC = NCC ? NCC : a.NC;  // columns (query x head) per slab; NCC: known at compile time
    const int T = nslab * NC;
    const int team = !FUSED || 2 * T > NW ? 1 : 3 * T > NW ? 2 : 3;  // warps a task
    int member = 0, first_task = warp;
    if (team > 1) {
        if (warp >= team * T) return;
        member = warp >= 2 * T ? 2 : warp >= T ? 1 : 0;
        first_task = warp - member * T;
    }
    // Tasks from the last: task t is (slab #si, column j); (si, j) go back by
    // subtractions: no division on this latency-bound path.
    int si = nslab - 1, j = NC - 1 - first_task;
#pragma unroll 1
    for (int t = T - 1 - first_task; t >= 0; t -= NW, j -= NW) {
#pragma unroll 1
        while (j < 0) {
            j += NC;
            --si;
        }
        unsigned m = fresh;
#pragma unroll 1
        for (int k = 0; k < si; ++k) m &= m - 1;
        const int e0 = uniform(__ffs(m) - 1);
        const int h = uniform(__shfl_sync(kFull, h_e, e0));
        const bool before = uniform(__shfl_sync(kFull, p0_e, e0) < A) != 0, after = uniform(__shfl_sync(kFull, p1_e, e0) > Bc) != 0;
        const bool merger = FUSED && before && !after;  // this CTA is the slab's last of several
        if (member > 0 && !merger) return;
        float M = -INFINITY, L = 0.f;
        float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
        if (member == 0) {
            // Lane e holds (m, l) of entry e when it is of this slab: odd entries in the
            // warps' rings, even ones (at most one in a CTA whose slabs are longer than a
            // warp's range) in the warp records.
            const unsigned same = __ballot_sync(kFull, h_e == h);
            const float* rf = reinterpret_cast<const float*>(ring);
            const int ring_floats = ring_bytes / 4;
            float2 ml = make_float2(-INFINITY, 0.f);
            if (h_e == h)
                ml = *reinterpret_cast<const float2*>(
                    (lane & 1) ? rf + (lane >> 1) * ring_floats + NC * kHeadDim + 2 * j
                               : a.warp_ml + (((int64_t)c * NW + (lane >> 1)) * NC + j) * 2);
            M = ml.x;
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) M = fmaxf(M, __shfl_xor_sync(kFull, M, o));
            const float f = (ml.x == -INFINITY) ? 0.f : ex2(ml.x - M);
            rf += j * kHeadDim + 4 * lane;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const float fw = __shfl_sync(kFull, f, 2 * w + 1);  // 0 when the entry is not of this slab
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if ((same >> (2 * w + 1)) & 1u) v = *reinterpret_cast<const float4*>(rf + w * ring_floats);
                O.x = fmaf(v.x, fw, O.x);
                O.y = fmaf(v.y, fw, O.y);
                O.z = fmaf(v.z, fw, O.z);
                O.w = fmaf(v.w, fw, O.w);
            }
#pragma unroll 1
            for (unsigned e = uniform(same & 0x55555555u); e; e &= e - 1) {
                const int w2 = __ffs(e) - 1;
                const float fw = __shfl_sync(kFull, f, w2);
                const float4 v = reinterpret_cast<const float4*>(
                    a.warp_o + (((int64_t)c * NW + (w2 >> 1)) * NC + j) * kHeadDim)[lane];
                O.x = fmaf(v.x, fw, O.x);
                O.y = fmaf(v.y, fw, O.y);
                O.z = fmaf(v.z, fw, O.z);
                O.w = fmaf(v.w, fw, O.w);
            }
            L = f * ml.y;
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) L += __shfl_xor_sync(kFull, L, o);
        }
        if (!FUSED) {
            const int64_t sj = ((int64_t)c + h) * NC + j;
            reinterpret_cast<float4*>(a.work_o + sj * kHeadDim)[lane] = O;
            if (lane == 0) *reinterpret_cast<float2*>(a.work_ml + sj * 2) = make_float2(M, L);
            continue;
        }
        if (after) {
            put_partial(a, c, j, NC, O, M, L, lane);
            continue;
        }
        bool good = true;
        if (merger) {
            float* dep = reinterpret_cast<float*>(ring + warp * ring_bytes + dep_off);
            if (team == 1 || member > 0)
                good = merge_partials<12, NCC>(a, j, NC, meta[TM::kC0] + max(member - 1, 0), team == 3 ? 2 : 1,
                                                   c + a.merge_extra, M, L, O, lane);
            if (member > 0) {
                reinterpret_cast<float4*>(dep)[lane] = O;
                if (lane == 0) *reinterpret_cast<float4*>(dep + kHeadDim) = make_float4(M, L, good ? 1.f : 0.f, 0.f);
                bar_arrive(1 + t, 32 * team);
                return;
            }
            if (team > 1) {
                bar_sync(1 + t, 32 * team);
#pragma unroll
                for (int k = 1; k <= 2; ++k) {
                    if (k >= team) break;
                    const float* d = dep + k * T * (ring_bytes / 4);
                    const float4 v = reinterpret_cast<const float4*>(d)[lane];
                    const float4 ml = *reinterpret_cast<const float4*>(d + kHeadDim);
                    good &= ml.z != 0.f;
                    const float Mb = fmaxf(M, ml.x);
                    const float f0 = (M == -INFINITY) ? 0.f : ex2(M - Mb), f1 = (ml.x == -INFINITY) ? 0.f : ex2(ml.x - Mb);
                    M = Mb;
                    L = fmaf(ml.y, f1, L * f0);
                    O.x = fmaf(v.x, f1, O.x * f0);
                    O.y = fmaf(v.y, f1, O.y * f0);
                    O.z = fmaf(v.z, f1, O.z * f0);
                    O.w = fmaf(v.w, f1, O.w * f0);
                }
            }
        }
        if (good) write_out<G>(a, h / a.Hkv, h % a.Hkv, j, O, L, lane);
    }
}

// Launch with programmatic stream serialization: the kernel may start while the
// previous kernel in the stream drains, and waits (griddepcontrol.wait) before
// it reads that kernel's results.
template <class K, class... Args>
cudaError_t launch_pdl(K kernel, int grid, int block, int smem, cudaStream_t st, const Args&... args)
{
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(block);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, kernel, args...);
}

}  // namespace
}  // namespace dkv
