// Decode-step attention over the packed cache (Sec. 3.4), split-K, with both
// contractions of a tile on the tensor cores.
//
// Work split, slab segments and merges are those of the fp32 kernel
// (dkv_decode_common.cuh). What differs is the tile: the K and the V rows of 16
// cache rows are a half-tile each, one 3-D TMA box (64 dims x 16 rows x the two
// 64-dim halves, 128-byte swizzle, so ldmatrix reads them without bank
// conflicts), and per tile the warp runs
//   S   = K q^T      8 x mma.sync m16n8k16 (bf16 in, fp32 accumulate): the 16
//                    rows are the M side, the G query heads of the KV head the
//                    n = 8 columns (heads G..7 are zero), two chains of four,
//   P   = 2^(S*scale*log2 e - m) with the lazily rescaled running max m,
//   O^T += V^T P^T   8 x 2 mma.sync: V^T via ldmatrix.trans, P^T via movmatrix;
//                    P enters as a bf16 high part plus a bf16 remainder, two
//                    products, which keeps about 16 significant bits of P.
// The query is already bf16 and K is bf16, so S is exact products summed in
// fp32, as in the fp32 kernel; only the summation order differs.
//
// The boxes read whole 16-row tiles even at the end of a segment: the rows past
// it (another slab's rows, reserve rows, or zero fill past the end of the cache)
// get score -inf and their V rows are zeroed in shared memory before use.
//
// What bounds a launch: HBM while it streams (a dense 128K layer runs at 0.98 of
// the copy rate), and around that about 5 us of latency: the first tiles after
// the previous kernel ends, and the merge after the last row. The work of those
// parts is scalar and runs once, so it is kept short: warp-uniform values are
// marked as such (without that every vote and shuffle carries a check for a
// split warp), rare code is out of line, nothing lives in a stack frame. Same-box
// us per step, 32 layers: 128K 1,065 -> 1,017, 32K 469 -> 422, 4K 312 -> 259; Qwen
// shape 64K x 4, 28 layers: 982 -> 919. (Rows appended by earlier calls, which are
// fetched only after the previous kernel, then cost 0.5 % at 128K and 1 % at 32K, with
// half of a reserve of 256 filled.)
#include "dkv_decode_common.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <math.h>

#include <mutex>
#include <type_traits>

namespace dkv {
namespace {

constexpr int kMmaTR = kBoxRows;          // rows per tile: the m16 of the score product, one TMA box
static_assert(kMmaTR == 16, "m16n8k16");
constexpr int kBoxBytes = kMmaTR * 128;   // one TMA box: 16 rows x 64 bf16 dims
constexpr int kHalfTile = 2 * kBoxBytes;  // the K (or V) rows of a tile: dims 0-63, then dims 64-127

template <int G, int NT, int NS_, int NW_>
struct MK {
    static constexpr int NS = NS_, NW = NW_, TR = kMmaTR;
    static constexpr int kWarpRing = NS * kHalfTile;
    static constexpr int kRingBytes = NW * kWarpRing;
    static constexpr int kBarBytes = NW * NS * 8;
    static constexpr int kMetaBytes = (TailMeta<NW>::kWords + kSegmentWords * NW) * 4;  // and a segment slot a warp
    static constexpr int kDepOff = (8 * NT * (kHeadDim + 2) * 4 + 15) / 16 * 16;  // after a warp's final state
    static constexpr int kAlign = 1024;                  // swizzle atoms are 1024-byte aligned
    static constexpr int kFixedBytes = kRingBytes + kBarBytes + kMetaBytes;
    static int bytes(int B, int NHl) { return kAlign + kFixedBytes + seq_table_bytes(B, NHl); }
    static_assert(NS >= 2, "a K and a V half-tile");
    static constexpr int kMaxBytes = kAlign + kFixedBytes + seq_table_bytes(kMaxB);  // the largest layer
    static_assert(kMaxBytes <= 227 * 1024, "fits the opt-in shared memory of one CTA");
    static_assert(kDepOff + 528 <= kWarpRing, "a warp's final state and a deposit fit in its ring");
};

// Half-tiles of a warp's ring, warps per CTA. One column tile (the decode step):
// more warps hide more of a tile's latency chain (score MMAs, softmax, output
// MMAs), and at the end of a pass the CTA's (slab, column) merge tasks spread
// over more warps, which counts for G > 4 (G tasks per slab). Multi-query with
// one column tile: Q G columns give up to 8 merge tasks per slab, so 16 warps.
// Two column tiles: twice the accumulators still fit 12 warps, and four half-
// tiles hold a 16-column final state.
//
// The ring holds 192 KB, one CTA per SM. Half of it (8 warps x 3 half-tiles or
// 10 and 12 x 2, two CTAs per SM, so that the next launch's CTAs are resident and
// have their first tiles before this launch ends) starts a launch sooner (first
// tile of the last CTA 0.4 instead of 4 us after the previous kernel) but streams
// slower per warp: 1,072, 1,120 and 1,222 against 1,017 us per step at 128K, 476,
// 508 and 625 against 422 at 32K, 248, 295 and 371 against 259 at 4K.
constexpr int kRingSmallG = 4, kWarpsSmallG = 12;
constexpr int kRingLargeG = 2, kWarpsLargeG = 16;
constexpr int kRingMulti1 = 2, kWarpsMulti1 = 16;
constexpr int kRingMulti2 = 4, kWarpsMulti2 = 12;
// Right after the wait for the previous kernel, a warp has one tile landed and
// one in flight: half its ring (or all of it, G > 4). The rows of its next tile
// are prefetched into L2 then, to fill the memory pipe while its first tiles are
// computed (us per step without -> with: Qwen shape 930 -> 919, 128K 1,018 ->
// 1,017). A warp with a short range gains nothing and its prefetches delay the
// copies its first tiles wait for, so only warps with at least kL2MinRows rows
// prefetch (prefetching in every warp cost 10 % at 32K, 54 rows a warp).
constexpr int kL2MinRows = 64;

template <int G, int NT, bool MULTI>
using MKFor = typename std::conditional<
    (NT > 1), MK<G, NT, kRingMulti2, kWarpsMulti2>,
    typename std::conditional<
        MULTI, MK<G, 1, kRingMulti1, kWarpsMulti1>,
        typename std::conditional<(G <= 4), MK<G, 1, kRingSmallG, kWarpsSmallG>,
                                  MK<G, 1, kRingLargeG, kWarpsLargeG>>::type>::type>::type;

// ------------------------------------------------------------ PTX wrappers
// The rows [row, row + 16) of a cache, both 64-dim halves (the map's dimensions:
// 64 dims, rows, halves).
__device__ __forceinline__ void tma_load_rows(uint32_t dst, const CUtensorMap* map, int row, uint32_t bar, uint64_t pol)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3, %2}], [%4], %5;" ::"r"(dst),
        "l"(map), "r"(0), "r"(row), "r"(bar), "l"(pol)
        : "memory");
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// d += a b, m16n8k16, bf16 operands, fp32 accumulators.
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t movm_t(uint32_t x)
{
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}

// bf16 pair (lo in the low half), round to nearest even.
__device__ __forceinline__ uint32_t bf16x2(float lo, float hi)
{
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// Byte offset of 16-byte chunk ch (0..7) of row r in a 128-byte-swizzled box.
__device__ __forceinline__ int swz(int r, int ch) { return r * 128 + ((ch ^ (r & 7)) << 4); }

// ------------------------------------------------------------ per-warp state
// Columns: the n side of both products, NT tiles of 8. Column c is query c / G,
// head c % G of the KV head's group (the decode step has one query: c = head).
// Lane (gid = lane / 4, t = lane % 4) holds columns 8 nt + 2t and 8 nt + 2t + 1.
template <int NT>
struct MmaState {
    float m[NT][2];     // running max of the two columns (log2 domain), the same in all gid lanes
    float l[NT][2];     // this lane's share of their softmax denominators
    float o[NT][8][4];  // O^T: [tile][dim block db][(dim 16 db + gid, col 2t), (.., 2t+1), (dim +8, 2t), (.., 2t+1)]
};

template <int NT>
__device__ __forceinline__ void state_reset(MmaState<NT>& S)
{
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        S.m[nt][0] = S.m[nt][1] = -INFINITY;
        S.l[nt][0] = S.l[nt][1] = 0.f;
#pragma unroll
        for (int db = 0; db < 8; ++db) S.o[nt][db][0] = S.o[nt][db][1] = S.o[nt][db][2] = S.o[nt][db][3] = 0.f;
    }
}

// q of the slab's columns as B fragments of the score product: for tile nt and k
// step kk (dims 16 kk .. 16 kk + 15), (column 8 nt + gid, dims 2t, 2t+1) and
// (column 8 nt + gid, dims 2t+8, 2t+9); zero past the last column.
template <int G, int NT>
__device__ __forceinline__ void load_q(const DecodeArgs& a, int b, int g, int NC, int lane, uint32_t (&qb)[NT][8][2])
{
    const int gid = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const int col = 8 * nt + gid;
        const bool live = col < NC;
        const int qi = col / G, j = col - qi * G;
        const uint32_t* qr =
            reinterpret_cast<const uint32_t*>(a.q + (live ? ((int64_t)b * a.Q + qi) * a.H + g * G + j : 0) * kHeadDim);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
            qb[nt][kk][0] = live ? ld_prev(qr + 8 * kk + t) : 0u;
            qb[nt][kk][1] = live ? ld_prev(qr + 8 * kk + t + 4) : 0u;
        }
    }
}

// Scores of one tile: stage holds its K rows.
template <int NT>
__device__ __forceinline__ void tile_scores(float (&c)[NT][4], const uint32_t (&qb)[NT][8][2], uint32_t stage, int lane)
{
    // Scores: ldmatrix lane -> (row, chunk) of the A fragment: rows 0-7 / 8-15 by
    // bit 3 of the lane, chunk +0 / +1 by bit 4. One K fragment serves all tiles.
    const int ar = (lane & 7) + (lane & 8), ac = lane >> 4;
    // Two chains of four products a tile: half the latency of one chain of eight.
    float c2[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) c[nt][i] = c2[nt][i] = 0.f;
    uint32_t af[8][4];
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) ldsm_x4(stage + (kk >> 2) * kBoxBytes + swz(ar, (kk & 3) * 2 + ac), af[kk]);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            mma16816(c[nt], af[kk], qb[nt][kk][0], qb[nt][kk][1]);
            mma16816(c2[nt], af[kk + 4], qb[nt][kk + 4][0], qb[nt][kk + 4][1]);
        }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) c[nt][i] += c2[nt][i];
}

// Softmax of one tile: the scores c become P^T as B fragments, a bf16 high part
// and remainder. Rows >= cnt are not part of the segment.
template <int NT>
__device__ __forceinline__ void tile_softmax(MmaState<NT>& S, const float (&c)[NT][4], uint32_t (&bh0)[NT],
                                             uint32_t (&bh1)[NT], uint32_t (&bl0)[NT], uint32_t (&bl1)[NT], int cnt,
                                             float cs, int lane)
{
    const int gid = lane >> 2;
    // c: (row gid, columns 2t, 2t+1), (row gid + 8, columns 2t, 2t+1). Lazy
    // rescaling as in the fp32 kernel: a column's running max only moves when a
    // score tops it by more than kSlack.
    float s[NT][4];
    bool over = false;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
        for (int i = 0; i < 4; ++i) s[nt][i] = c[nt][i] * cs;
        if (gid >= cnt) s[nt][0] = s[nt][1] = -INFINITY;
        if (gid + 8 >= cnt) s[nt][2] = s[nt][3] = -INFINITY;
        over |= fmaxf(s[nt][0], s[nt][2]) > S.m[nt][0] + kSlack || fmaxf(s[nt][1], s[nt][3]) > S.m[nt][1] + kSlack;
    }
    if (__any_sync(kFull, over)) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            float y0 = fmaxf(s[nt][0], s[nt][2]), y1 = fmaxf(s[nt][1], s[nt][3]);
#pragma unroll
            for (int o = 4; o <= 16; o <<= 1) {
                y0 = fmaxf(y0, __shfl_xor_sync(kFull, y0, o));
                y1 = fmaxf(y1, __shfl_xor_sync(kFull, y1, o));
            }
            const float mn0 = fmaxf(S.m[nt][0], y0), mn1 = fmaxf(S.m[nt][1], y1);
            const float al0 = (mn0 == -INFINITY) ? 1.f : ex2(S.m[nt][0] - mn0);
            const float al1 = (mn1 == -INFINITY) ? 1.f : ex2(S.m[nt][1] - mn1);
            S.l[nt][0] *= al0;
            S.l[nt][1] *= al1;
#pragma unroll
            for (int db = 0; db < 8; ++db) {
                S.o[nt][db][0] *= al0;
                S.o[nt][db][1] *= al1;
                S.o[nt][db][2] *= al0;
                S.o[nt][db][3] *= al1;
            }
            S.m[nt][0] = mn0;
            S.m[nt][1] = mn1;
        }
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const float r0 = (S.m[nt][0] == -INFINITY) ? 0.f : S.m[nt][0];
        const float r1 = (S.m[nt][1] == -INFINITY) ? 0.f : S.m[nt][1];
        const float p0 = ex2(s[nt][0] - r0), p1 = ex2(s[nt][1] - r1);  // 2^-inf = 0
        const float p2 = ex2(s[nt][2] - r0), p3 = ex2(s[nt][3] - r1);
        S.l[nt][0] += p0 + p2;
        S.l[nt][1] += p1 + p3;
        // P^T as B fragments: bf16 high part and remainder, transposed by movmatrix
        // from (row, column pair) to (row pair, column).
        const uint32_t h01 = bf16x2(p0, p1), h23 = bf16x2(p2, p3);
        const uint32_t l01 = bf16x2(p0 - __uint_as_float(h01 << 16), p1 - __uint_as_float(h01 & 0xffff0000u));
        const uint32_t l23 = bf16x2(p2 - __uint_as_float(h23 << 16), p3 - __uint_as_float(h23 & 0xffff0000u));
        bh0[nt] = movm_t(h01);
        bh1[nt] = movm_t(h23);
        bl0[nt] = movm_t(l01);
        bl1[nt] = movm_t(l23);
    }
}

// The tile's share of the outputs: stage holds its V rows (zero past the segment).
template <int NT>
__device__ __forceinline__ void tile_output(MmaState<NT>& S, const uint32_t (&bh0)[NT], const uint32_t (&bh1)[NT],
                                            const uint32_t (&bl0)[NT], const uint32_t (&bl1)[NT], uint32_t stage,
                                            int lane)
{
    // O^T += V^T P^T: ldmatrix.trans lane -> (row, chunk): rows 0-7 / 8-15 by
    // bit 4 of the lane, chunk +0 / +1 by bit 3. One V fragment serves all tiles.
    const int vr = (lane & 7) + ((lane >> 4) << 3), vc = (lane >> 3) & 1;
    // Four fragments at a time, their products in an order that keeps a column
    // block's two products four apart.
#pragma unroll
    for (int d0 = 0; d0 < 8; d0 += 4) {
        uint32_t af[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            ldsm_x4_t(stage + (d0 >> 2) * kBoxBytes + swz(vr, i * 2 + vc), af[i]);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
            for (int i = 0; i < 4; ++i) mma16816(S.o[nt][d0 + i], af[i], bh0[nt], bh1[nt]);
#pragma unroll
            for (int i = 0; i < 4; ++i) mma16816(S.o[nt][d0 + i], af[i], bl0[nt], bl1[nt]);
        }
    }
}

// Softmax denominators of the lane's columns, summed over the gid lanes.
template <int NT>
__device__ __forceinline__ void finish_l(const MmaState<NT>& S, float (&l2)[NT][2])
{
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        float a = S.l[nt][0], b = S.l[nt][1];
#pragma unroll
        for (int o = 4; o <= 16; o <<= 1) {
            a += __shfl_xor_sync(kFull, a, o);
            b += __shfl_xor_sync(kFull, b, o);
        }
        l2[nt][0] = a;
        l2[nt][1] = b;
    }
}

// The state, scaled by f, into rows of 128 floats: column c at o_dst + (c / G) *
// q_stride + (c % G) * 128 (a record's columns follow each other: q_stride =
// G * 128), and (m, l)[NC] at ml_dst unless that is null. One copy serves the
// warp's ring, its record, a workspace slot and the output (generic stores).
template <int G, int NT>
__device__ __forceinline__ void store_mma_state(const MmaState<NT>& S, const float (&f)[NT][2],
                                                const float (&l2)[NT][2], float* o_dst, int q_stride, float* ml_dst,
                                                int NC, int lane)
{
    const int gid = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int j = 8 * nt + 2 * t + q;
            if (j < NC) {
                const int qi = j / G;
                float* dst = o_dst + qi * q_stride + (j - qi * G) * kHeadDim + gid;
#pragma unroll
                for (int db = 0; db < 8; ++db) {
                    dst[16 * db] = S.o[nt][db][q] * f[nt][q];
                    dst[16 * db + 8] = S.o[nt][db][2 + q] * f[nt][q];
                }
                if (ml_dst && gid == 0) *reinterpret_cast<float2*>(ml_dst + 2 * j) = make_float2(S.m[nt][q], l2[nt][q]);
            }
        }
}

// ------------------------------------------------------------ rarely run parts
// These run a few times a launch at most. They are functions of their own so
// that the kernel's code stays short and its registers stay with the tile loop.

// This step's key (value: the upper 16 lanes') row, 16 bytes a lane: into the tile
// at st, as its row `row`, and into the cache at dst for later steps (null: not).
__device__ __noinline__ void append_row(unsigned char* st, int row, uint4 v, uint16_t* dst, bool value, int lane)
{
    const int sub = lane & 15;
    if ((lane >> 4) == (value ? 1 : 0)) {
        *reinterpret_cast<uint4*>(st + (sub >> 3) * kBoxBytes + swz(row, sub & 7)) = v;
        if (dst) *(reinterpret_cast<uint4*>(dst) + sub) = v;
    }
    fence_proxy_async_smem();  // order these generic writes before later bulk copies
    __syncwarp();
}

// V rows [cnt, 16) of a tile, past its segment: zeros (their p is 0, but 0 * inf
// or 0 * nan would not be).
__device__ __noinline__ void zero_rows(unsigned char* st, int cnt, int lane)
{
#pragma unroll 1
    for (int k = lane; k < (kMmaTR - cnt) * 16; k += 32) {
        const int row = cnt + (k >> 4), sub = k & 15;
        *reinterpret_cast<uint4*>(st + (sub >> 3) * kBoxBytes + swz(row, sub & 7)) = make_uint4(0u, 0u, 0u, 0u);
    }
    fence_proxy_async_smem();  // order these generic writes before later bulk copies
    __syncwarp();
}

// The CTA that holds the first row of the slab of layer row A.
__device__ __noinline__ void first_cta(const DecodeArgs& a, unsigned char* table, int A, int R, int P, int32_t* out)
{
    const SeqTable t = seq_table_at(table, a);
    *out = part_of(slab_start(a, t, slab_containing(a, t, a.B * a.Hkv, A)), R, P);
}

// Slabs with no rows belong to no CTA: their outputs are zero.
template <int G>
__device__ __noinline__ void write_empty_slabs(const DecodeArgs& a, unsigned char* table, int NC, int lane)
{
    const SeqTable t = seq_table_at(table, a);
#pragma unroll 1
    for (int h = 0; h < a.B * a.Hkv; ++h)
        if (slab_start(a, t, h) == slab_start(a, t, h + 1))
#pragma unroll 1
            for (int j = 0; j < NC; ++j)
                write_out<G>(a, h / a.Hkv, h % a.Hkv, j, make_float4(0.f, 0.f, 0.f, 0.f), 0.f, lane);
}

// ------------------------------------------------------------ kernel
// MULTI: columns are Q x G with Q from the arguments (multi-query); otherwise
// the G heads of the decode step, fixed at compile time.
template <int G, int NT, bool FUSED, bool MULTI>
__global__ void __launch_bounds__(MKFor<G, NT, MULTI>::NW * 32, 1)
    decode_mma_kernel(const __grid_constant__ DecodeArgs a, const __grid_constant__ CacheMaps maps)
{
    using C = MKFor<G, NT, MULTI>;
    constexpr int NCC = MULTI ? 0 : G;
    const int NC = MULTI ? a.NC : G;
    constexpr int TR = C::TR, NS = C::NS, NW = C::NW;
    // Half-tiles fetched before the wait for the previous kernel: they compete with its
    // merge, and fill the memory pipe while it runs (us per step with 2, 3, 4: 128K
    // 1,018 / 1,007 / 1,033, 32K 425 / 423 / 461, ragged batch of 16 662 / 655 / 656).
    constexpr int NPRE = NS < 3 ? NS : 3;
    static_assert(NPRE <= 3, "the first two tiles are checked for rows that an earlier call appends");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // The ring starts on a 1024-byte boundary (the swizzle pattern's period).
    unsigned char* smem = smem_raw + ((C::kAlign - (smem_u32(smem_raw) & (C::kAlign - 1))) & (C::kAlign - 1));
    unsigned char* table = smem + C::kFixedBytes;
    const SeqTable tab = seq_table_at(table, a);
    using TM = TailMeta<NW>;
    int32_t* meta = reinterpret_cast<int32_t*>(smem + C::kRingBytes + C::kBarBytes);

    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int NHl = a.B * a.Hkv;
    const int c = blockIdx.x;
    uint64_t* my_bars = reinterpret_cast<uint64_t*>(smem + C::kRingBytes) + warp * NS;

    if (warp == 0)
        build_seq_table(a, tab, c == 0);
    else
        load_slab_cache(a, tab, 32, (NW - 1) * 32);
    if (lane == 0) {
#pragma unroll 1
        for (int s = 0; s < NS; ++s) mbar_init(smem_u32(&my_bars[s]), 1);
        fence_proxy_async_smem();
        meta[TM::kFirst + warp] = -1;
        meta[TM::kLast + warp] = -1;
        if (warp == 0) meta[TM::kDead] = 0;
    }
    __syncthreads();  // table, barriers and slab entries are ready
    finish_slab_cache(a, tab, NW * 32);
    __syncthreads();

    const int R = uniform(slab_start(a, tab, NHl));
    if (FUSED && c == a.nctas - 1 && warp == 0) {
        // Written by the last CTA, which always runs; after the wait, as any write of out.
        pdl_wait();
        write_empty_slabs<G>(a, table, NC, lane);
    }
    const int P = live_parts(R, a.nctas);  // CTAs with rows
    const int A = c < P ? part_start(c, R, P) : R, Bc = c < P ? part_start(c + 1, R, P) : R;
    if (A >= Bc) {  // uniform: this CTA has no rows
        pdl_wait();
        return;
    }
    const int wA = A + (int)(((int64_t)(Bc - A) * warp) / NW);
    const int wB = A + (int)(((int64_t)(Bc - A) * (warp + 1)) / NW);
    unsigned char* my_ring = smem + warp * C::kWarpRing;
    // First CTA of the CTA's first slab, for the end of the pass.
    if (FUSED && warp == NW - 1) first_cta(a, table, A, R, P, meta + TM::kC0);
    MmaState<NT> S;
    float l2[NT][2];

    if (wA < wB) {
        const int2 hr = slab_range(a, table, wA, wB);
        const int hfirst = uniform(hr.x), hlast = uniform(hr.y);
        const uint64_t pol = evict_first_policy();
        int32_t* slot = meta + TM::kWords + kSegmentWords * warp;
        find_segment(a, table, hfirst, hlast + 1, wA, wB, slot);
        Segment cp = read_segment(slot);  // the segment being computed; `left` and `row` run on tile by tile
        int ld_h = cp.h, ld_left = cp.left, ld_row = cp.row;  // the next tile to fetch

        // Half-tiles stream through the warp's ring in the order K0 V0 K1 V1 ...
        // Whole 16-row boxes from the tile's first cache row; the rows past the
        // segment are masked later. (The new token's row is read too and then
        // overwritten in shared memory from k_new / v_new.)
        int vrow = -1;  // cache row of the tile whose V half is the next to issue; -1: a K half is
        int fill = 0;   // slot of the next half-tile to issue
        int inflight = 0;
        auto issue_next = [&]() {
            const bool is_v = vrow >= 0;
            if (!is_v && ld_left <= 0) return;
            const int row = is_v ? vrow : ld_row;
            if (lane == 0) {
                // Bounds-checked build: the tile's rows lie in the cache (a TMA box past
                // the end reads zeros, so the copy itself stays in bounds either way).
                in_bounds(row >= 0 && (is_v || a.rows_cap == 0 || row + min(TR, ld_left) <= a.rows_cap), a.status);
                const uint32_t bar = smem_u32(&my_bars[fill]);
                mbar_arrive_expect_tx(bar, kHalfTile);
                tma_load_rows(smem_u32(my_ring + fill * kHalfTile), is_v ? &maps.v : &maps.k, row, bar, pol);
            }
            ++inflight;
            if (++fill == NS) fill = 0;
            if (is_v) {
                vrow = -1;
                return;
            }
            vrow = row;
            ld_row += TR;
            ld_left -= TR;
            if (ld_left <= 0 && ld_h < hlast) {
                find_segment(a, table, ld_h + 1, hlast + 1, wA, wB, slot);
                ld_h = uniform(slot[0]);
                ld_left = uniform(slot[1]);
                ld_row = uniform(slot[2]);
            }
        };

        // A bounded wait that runs out marks the warp dead: it stops issuing and
        // computing, drains its copies in flight, and leaves its partials unwritten.
        bool dead = false;
        // Before the wait, only tiles of settled rows (K0 V0 K1: the first two tiles).
        const int whole = cp.settled >= cp.left ? NPRE : 2 * (cp.settled / TR);
        int pre = 0;
#pragma unroll 1
        for (; pre < min(NPRE, whole); ++pre) {
            // A second tile of another segment, which is then the one in the slot.
            if (pre == 2 && cp.left <= TR && uniform(slot[6]) < min(TR, ld_left)) break;
            issue_next();
        }
        // Everything above reads only the plan, n_appended and context rows; rows
        // appended by earlier calls, q, k_new, v_new, the cache slots written here and
        // the workspace belong to the previous kernel's epoch.
        pdl_wait();
        pdl_launch_dependents();  // only now: the next kernel may then rely on everything before this one
#pragma unroll 1
        for (int s = pre; s < NS; ++s) issue_next();
        int stage = 0;
        uint32_t phase = 0;
        const float cs = a.qscale;  // softmax scale * log2(e)
        bool prefetch = wB - wA >= kL2MinRows;

#pragma unroll 1
        for (;;) {
            const int h = cp.h;
            const int b = h / a.Hkv, g = h - b * a.Hkv;
            uint32_t qb[NT][8][2];
            load_q<G, NT>(a, b, g, NC, lane, qb);
            // This step's row, if the segment ends with it: k_new in lanes 0-15, v_new in
            // 16-31, requested with q (its tile is on the way to the slab's merge: two
            // round trips there held up every slab by 1.4 us).
            uint4 fresh_row = make_uint4(0u, 0u, 0u, 0u);
            if (cp.app)
                fresh_row = ld_prev(reinterpret_cast<const uint4*>((lane < 16 ? a.k_new : a.v_new) +
                                                                 ((int64_t)b * a.Hkv + g) * kHeadDim) + (lane & 15));
            state_reset(S);
            if (prefetch) {
                // The next tile's K and V rows into L2: exactly the segment's rows, all in the cache.
                prefetch = false;
                if (lane == 0 && ld_left > 0) {
                    const uint32_t bytes = (uint32_t)min(TR, ld_left) * kRowBytes;
                    prefetch_l2_bulk(a.Kc + (int64_t)ld_row * kHeadDim, bytes);
                    prefetch_l2_bulk(a.Vc + (int64_t)ld_row * kHeadDim, bytes);
                }
            }

#pragma unroll 1
            while (cp.left > 0) {
                const int cnt = min(TR, cp.left);
                const bool newest = cp.app && cp.left <= TR;  // the tile holds this step's token
                const int64_t new_row = cp.row + cnt - 1;
                const bool new_ok = newest && in_bounds(a.rows_cap == 0 || new_row < a.rows_cap, a.status);
                float sc[NT][4];
                {
                    unsigned char* st = my_ring + stage * kHalfTile;
                    // Every lane observes the completed phase itself (acquire) before reading.
                    if (!__all_sync(kFull, mbar_wait(smem_u32(&my_bars[stage]), phase))) {
                        dead = true;
                        break;
                    }
                    --inflight;
                    if (newest)
                        append_row(st, cnt - 1, fresh_row, new_ok ? a.Kc + new_row * kHeadDim : nullptr, false, lane);
                    tile_scores<NT>(sc, qb, smem_u32(st), lane);
                    __syncwarp();
                    if (++stage == NS) {
                        stage = 0;
                        phase ^= 1u;
                    }
                    issue_next();  // into the K half's slot
                }
                uint32_t bh0[NT], bh1[NT], bl0[NT], bl1[NT];
                tile_softmax<NT>(S, sc, bh0, bh1, bl0, bl1, cnt, cs, lane);
                unsigned char* st = my_ring + stage * kHalfTile;
                if (!__all_sync(kFull, mbar_wait(smem_u32(&my_bars[stage]), phase))) {
                    dead = true;
                    break;
                }
                --inflight;
                if (newest)
                    append_row(st, cnt - 1, fresh_row, new_ok ? a.Vc + new_row * kHeadDim : nullptr, true, lane);
                if (cnt < TR) zero_rows(st, cnt, lane);
                tile_output<NT>(S, bh0, bh1, bl0, bl1, smem_u32(st), lane);
                __syncwarp();
                if (++stage == NS) {
                    stage = 0;
                    phase ^= 1u;
                }
                issue_next();  // into the V half's slot
                cp.left -= TR;
                cp.row += TR;
            }
            if (dead) break;
            finish_l(S, l2);
            const bool last = h == hlast, first = h == hfirst;
            if (last || first) {
                if (lane == 0) {
                    meta[(last ? TM::kLast : TM::kFirst) + warp] = h;
                    meta[TM::kP0 + 2 * warp + (last ? 1 : 0)] = cp.p0;
                    meta[TM::kP1 + 2 * warp + (last ? 1 : 0)] = cp.p1;
                }
            }
            // The last slab's state goes to the warp's own ring, idle now (every tile it
            // issued was consumed), to be merged with the other warps'; the first's, which
            // continues in an earlier warp, to the warp's record; a slab in between lies
            // wholly in this warp's range and is the output itself (or the CTA's partial).
            const int64_t rec = last || first ? (int64_t)c * NW + warp : (int64_t)c + h;
            float* o_dst = last    ? reinterpret_cast<float*>(my_ring)
                           : first ? a.warp_o + rec * NC * kHeadDim
                           : FUSED ? a.out + out_row<G>(a, b, g, 0) * kHeadDim
                                   : a.work_o + rec * NC * kHeadDim;
            float* ml_dst = last    ? o_dst + NC * kHeadDim
                            : first ? a.warp_ml + rec * NC * 2
                            : FUSED ? nullptr
                                    : a.work_ml + rec * NC * 2;
            const bool to_out = FUSED && !last && !first;
            float f[NT][2];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int q = 0; q < 2; ++q) f[nt][q] = !to_out ? 1.f : l2[nt][q] > 0.f ? 1.f / l2[nt][q] : 0.f;
            __syncwarp();
            store_mma_state<G, NT>(S, f, l2, o_dst, MULTI && to_out ? a.H * kHeadDim : G * kHeadDim, ml_dst, NC, lane);
            if (last) break;
            find_segment(a, table, h + 1, hlast + 1, wA, wB, slot);
            cp = read_segment(slot);
        }

        if (dead && lane == 0) {
            // After a timeout, wait (with the same bound) for the copies still in flight.
            atomicOr(a.status, 0x2 /* DKV_DEV_TMA_TIMEOUT */);
            meta[TM::kDead] = 1;
#pragma unroll 1
            for (int k = 0; k < inflight; ++k) {
                mbar_wait(smem_u32(&my_bars[stage]), phase);
                if (++stage == NS) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
    } else {
        pdl_wait();
        pdl_launch_dependents();
    }
    // Then the CTA merges, all warps sharing the work.
    __syncthreads();
    if (FUSED && uniform(meta[TM::kDead])) {
        dead_tail<NW>(a, tab, NC, c, A, Bc, R, P, warp, lane);
        return;
    }
    cta_tail<G, NW, FUSED, NCC>(a, smem, C::kWarpRing, C::kDepOff, meta, c, A, Bc, warp, lane);
}

template <int G, int NT, bool FUSED, bool MULTI>
cudaError_t launch_mma_g(const DecodeArgs& a, const CacheMaps& maps, const DecodeConfig& cfg, cudaStream_t st)
{
    using C = MKFor<G, NT, MULTI>;
    // The configuration must be this kernel's: its warps and shared-memory layout;
    // the grid is the call's CTA count (at most the configuration's).
    if (cfg.nwarps != C::NW || cfg.smem_bytes < C::bytes(a.B, a.B * a.Hkv) || a.nctas < 1 || a.nctas > cfg.nctas)
        return cudaErrorInvalidConfiguration;
    return launch_pdl(decode_mma_kernel<G, NT, FUSED, MULTI>, a.nctas, C::NW * 32, cfg.smem_bytes, st, a, maps);
}

// Launch configuration of the tensor-core kernels of one kind: the decode step
// (NT = 1, partial and fused), or multi-query with NT column tiles (fused only).
template <int G, int NT, bool MULTI>
cudaError_t config_mma_g(int B, int NHl, DecodeConfig* cfg)
{
    using C = MKFor<G, NT, MULTI>;
    const int smem = C::bytes(B, NHl);
    cudaError_t e;
    // The attribute is the kernel's, not the plan's: always the most any plan needs, so
    // that plans of other sizes keep working beside each other.
    if constexpr (!MULTI) {
        if ((e = cudaFuncSetAttribute(decode_mma_kernel<G, NT, false, false>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, C::kMaxBytes)) != cudaSuccess)
            return e;
    }
    if ((e = cudaFuncSetAttribute(decode_mma_kernel<G, NT, true, MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  C::kMaxBytes)) != cudaSuccess)
        return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, decode_mma_kernel<G, NT, true, MULTI>, C::NW * 32,
                                                           smem)) != cudaSuccess)
        return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    cfg->nctas = sms;
    cfg->nwarps = C::NW;
    cfg->smem_bytes = smem;
    return cudaSuccess;
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

}  // namespace

cudaError_t make_cache_maps(const void* Kc, const void* Vc, int64_t rows, CacheMaps* maps, bool short_boxes,
                            int box_rows, bool halves)
{
    if (box_rows < 8 || box_rows > 256 || (box_rows & 7)) return cudaErrorInvalidValue;
    if (rows < 1 || rows > kMaxMmaRows) return cudaErrorInvalidValue;
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    // halves: 64 dims x rows x the two 64-dim halves of a row, so that one box
    // brings both halves of its rows, half after half.
    const cuuint64_t dim[3] = {(cuuint64_t)(halves ? 64 : kHeadDim), (cuuint64_t)rows, 2};
    const cuuint64_t stride[2] = {(cuuint64_t)kRowBytes, 128};
    // short_boxes (fault injection): 8-row boxes deliver half the bytes each
    // stage's mbarrier expects, inside the stage, so every wait runs out.
    const cuuint32_t box[3] = {64, (cuuint32_t)(short_boxes ? box_rows / 2 : box_rows), 2};
    const cuuint32_t elem[3] = {1, 1, 1};
    const void* base[2] = {Kc, Vc};
    CUtensorMap* out[2] = {&maps->k, &maps->v};
#pragma unroll 1
    for (int i = 0; i < 2; ++i)
        if (enc(out[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, halves ? 3 : 2, const_cast<void*>(base[i]), dim, stride, box, elem,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    return cudaSuccess;
}

cudaError_t decode_config_mma(int G, int B, int Hkv, int kind, DecodeConfig* cfg)
{
    const int NHl = B * Hkv;
    if (B < 1 || B > kMaxB || Hkv < 1 || kind < 0 || kind > 2) return cudaErrorInvalidValue;
#define DKV_CFG_CASE(g)                                                               \
    case g:                                                                           \
        return kind == 0 ? config_mma_g<g, 1, false>(B, NHl, cfg)                          \
                         : (kind == 1 ? config_mma_g<g, 1, true>(B, NHl, cfg) : config_mma_g<g, 2, true>(B, NHl, cfg));
    switch (G) {
        DKV_CFG_CASE(1)
        DKV_CFG_CASE(2)
        DKV_CFG_CASE(3)
        DKV_CFG_CASE(4)
        DKV_CFG_CASE(5)
        DKV_CFG_CASE(6)
        DKV_CFG_CASE(7)
        DKV_CFG_CASE(8)
        default: return cudaErrorInvalidValue;
    }
#undef DKV_CFG_CASE
}

template <bool FUSED>
static cudaError_t launch_mma_any(const DecodeArgs& a, const CacheMaps& maps, const DecodeConfig& cfg, cudaStream_t st)
{
    // The decode step (Q = 1) takes the kernels with the G columns fixed at
    // compile time; multi-query calls the fused ones with one or two column tiles.
    const bool multi = a.Q > 1, two = a.NC > 8;
    if (multi && !FUSED) return cudaErrorInvalidValue;
#define DKV_LAUNCH_CASE(g)                                                                        \
    case g:                                                                                       \
        return !multi ? launch_mma_g<g, 1, FUSED, false>(a, maps, cfg, st)                        \
                      : (two ? launch_mma_g<g, 2, true, true>(a, maps, cfg, st)                   \
                             : launch_mma_g<g, 1, true, true>(a, maps, cfg, st));
    switch (a.G) {
        DKV_LAUNCH_CASE(1)
        DKV_LAUNCH_CASE(2)
        DKV_LAUNCH_CASE(3)
        DKV_LAUNCH_CASE(4)
        DKV_LAUNCH_CASE(5)
        DKV_LAUNCH_CASE(6)
        DKV_LAUNCH_CASE(7)
        DKV_LAUNCH_CASE(8)
        default: return cudaErrorInvalidValue;
    }
#undef DKV_LAUNCH_CASE
}

cudaError_t launch_decode_mma_partial(const DecodeArgs& a, const CacheMaps& maps, const DecodeConfig& cfg,
                                      cudaStream_t st)
{
    return launch_mma_any<false>(a, maps, cfg, st);
}

cudaError_t launch_decode_mma_fused(const DecodeArgs& a, const CacheMaps& maps, const DecodeConfig& cfg,
                                    cudaStream_t st)
{
    return launch_mma_any<true>(a, maps, cfg, st);
}

}  // namespace dkv
