// Work split of the sweep kernels: "column threads" for everything elementwise on a 64-token tile and
// "split accumulators" for everything that comes back from tensor memory.
//
// Column threads.  256 threads; warp g owns rows 8 g .. 8 g + 7 of the tile (8 rows are also the shortest
// sub-chunk, so a warp's rows always share one centring) and a lane one pair of neighbouring channels of
// all 8 rows.  Its gates, their running sum, the decay factors and the operand rows stay in its registers
// from the global load to the fp16 store; the only thing that crosses warps is one sum per 8-row group
// and channel.  At d = 72 the four pairs beyond channel 64 are spread over the warp as one more item per
// lane (row lane / 4, pair 32 + lane % 4) whose sums are formed by shuffles; 288 threads with one pair each
// were measured against it: nine warps cannot be spread evenly over the four schedulers, which costs a
// quarter of the registers and spills.
// The split this replaces (one 8-channel chunk of one row per thread, gates through a shared fp32 table
// that was written, scanned in place and read back) executed 7.8 K (d = 64) and 12.2 K (d = 72) warp
// instructions per tile in the forward sweep, half of them address, predicate and table traffic.
// A warp's 32 pairs of a row are 128 contiguous bytes of bf16 and 256 of gates; 4-byte stores into the
// chunk-major tiles hit 32 different banks.  Every warp sees all channels, so decisions about a tile are
// warp votes over identical numbers and need no barrier.
//
// Split accumulators.  An M = 64 product fills lanes 0-15 of each tensor-memory lane quarter.  Products
// whose N side can be cut in two put the second half into lanes 16-31 of the same columns, so that all
// lanes of a tcgen05.ld carry data: value channels are cut at chunk NV0, score columns into even and odd
// 8-token chunks (which keeps the causal halves balanced).  At d = 72 the state product has 8 more key
// channels than M = 64 holds: that corner is computed transposed (value channels along M, 8 key
// channels along N) by the warps that own fewer value chunks.
#pragma once

#include "sweep.cuh"

namespace dig {
namespace sw {

template <int D>
struct Col {
    using C = Cfg<D>;
    static constexpr int NT = 256;
    static constexpr int NV0 = (C::NCH + 1) / 2, NV1 = C::NCH - NV0;   // value chunks in lanes 0-15 / 16-31
    static constexpr int HW = 8 * NV0;                  // accumulator columns of a product split by value chunks
    static constexpr bool X = D > 64;                   // more than 64 channels: extra items and a transposed corner
    static constexpr int ACCS = HW + (X ? 8 : 0);       // accumulator columns of a state product
    static constexpr int NPS = X ? 3 : 2;               // state pieces of 8 values per thread
    static constexpr int NPO = (NV0 + 1) / 2;           // output pieces per thread
    static_assert(T / kMinSub * 32 == NT, "a warp's rows are the shortest sub-chunk");
    static_assert(D == 64 || D == 72, "32 channel pairs, or 36 of which 4 are extra items");
};

__device__ __forceinline__ float2 ex2_2(float2 x) { return make_float2(ex2(x.x), ex2(x.y)); }
__device__ __forceinline__ float2 ex2_neg2(float2 x) { return make_float2(ex2(-x.x), ex2(-x.y)); }

// Rows of the tensors a kernel needs, 8 (+ the extra item) per thread.  g: the gates; later (log2 units) sums of them.
template <int D, bool HQ, bool HD>
struct Cols {
    static constexpr int N = Col<D>::X ? 9 : 8;          // item 8: the extra one
    uint32_t k[N], v[N], q[HQ ? N : 1], d[HD ? N : 1];
    float2 g[N];
};

// What a thread works on.
template <int D>
struct Who {
    int grp, c2;            // row group (warp), first channel of the pair
    int xrow, xc2;          // extra item: row inside the group, first channel
    int q4, cg, hf, r16;    // tensor-memory lane quarter, warp of the quarter (0 / 1), lane half, accumulator row (M = 64)
    // The last warp issues the MMAs and the bulk copies (under elect_one()).
    __device__ __forceinline__ bool issuer() const { return grp == Col<D>::NT / 32 - 1; }
    __device__ __forceinline__ Who()
    {
        const int lane = threadIdx.x & 31;
        grp = (int)warp_uniform(threadIdx.x >> 5);
        c2 = 2 * lane;
        xrow = lane >> 2;
        xc2 = 64 + 2 * (lane & 3);
        q4 = grp & 3;
        cg = grp >> 2;
        hf = lane >> 4;
        r16 = 16 * q4 + (lane & 15);
    }
};

// Element offsets of the thread's items (row + pair), from the tile's row-offset table.
template <int D>
__device__ __forceinline__ void row_offsets(const int *tab, const Who<D> &w, uint32_t (&off)[9])
{
    const int4 a = reinterpret_cast<const int4 *>(tab)[2 * w.grp], b = reinterpret_cast<const int4 *>(tab)[2 * w.grp + 1];
    const int r[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int j = 0; j < 8; ++j) off[j] = (uint32_t)(r[j] + w.c2);
    off[8] = Col<D>::X ? (uint32_t)(tab[8 * w.grp + w.xrow] + w.xc2) : 0u;
}
__device__ __forceinline__ uint32_t ldg4(const bf16 *p) { return __ldg(reinterpret_cast<const uint32_t *>(p)); }

template <int N>
__device__ __forceinline__ void load_gates(float2 (&g)[N], const float *gate, const uint32_t (&off)[9])
{
#pragma unroll
    for (int j = 0; j < N; ++j) g[j] = __ldg(reinterpret_cast<const float2 *>(gate + off[j]));
}
template <int D, bool HQ, bool HD>
__device__ __forceinline__ void load_rows(Cols<D, HQ, HD> &r, const bf16 *q, const bf16 *k, const bf16 *v, const bf16 *d_out,
                                          const uint32_t (&off)[9])
{
#pragma unroll
    for (int j = 0; j < r.N; ++j) {
        r.k[j] = ldg4(k + off[j]);
        r.v[j] = ldg4(v + off[j]);
        if (HQ) r.q[j] = ldg4(q + off[j]);
        if (HD) r.d[j] = ldg4(d_out + off[j]);
    }
}
// Asks the L2 for the warp's 8 rows of every tensor of a tile further ahead than the register prefetch
// reaches: four lanes per row, one 32-byte sector each per instruction.
template <int D, bool HQ, bool HD>
__device__ __forceinline__ void prefetch_rows(const bf16 *q, const bf16 *k, const bf16 *v, const bf16 *d_out, const int *tab, const Who<D> &w)
{
    const uint32_t o = (uint32_t)tab[8 * w.grp + w.xrow], l = threadIdx.x & 3;
#pragma unroll
    for (int i = 0; i < (2 * D + 127) / 128; ++i)
        if (i == 0 || l == 0) {
            const uint32_t e = o + 16 * l + 64 * i;
            prefetch_l2(k + e);
            prefetch_l2(v + e);
            if (HQ) prefetch_l2(q + e);
            if (HD) prefetch_l2(d_out + e);
        }
}
template <int D>
__device__ __forceinline__ void prefetch_gates(const float *gate, const int *tab, const Who<D> &w)
{
    const uint32_t o = (uint32_t)tab[8 * w.grp + w.xrow], l = threadIdx.x & 3;
#pragma unroll
    for (int i = 0; i < (4 * D + 127) / 128; ++i)
        if (8 * l + 32 * i < D) prefetch_l2(gate + o + 8 * l + 32 * i);
}
template <int D> __device__ __forceinline__ int item_row(const Who<D> &w, int j) { return 8 * w.grp + (j < 8 ? j : w.xrow); }
// Rows past the end of the sequence (last tile only): zero operands.
template <int D, bool HQ, bool HD>
__device__ __forceinline__ void clear_tail_rows(Cols<D, HQ, HD> &r, const Who<D> &w, int nrow)
{
#pragma unroll
    for (int j = 0; j < r.N; ++j)
        if (item_row(w, j) >= nrow) {
            r.k[j] = r.v[j] = 0u;
            if (HQ) r.q[j] = 0u;
            if (HD) r.d[j] = 0u;
        }
}
template <int D, bool HQ, bool HD>
__device__ __forceinline__ void clear_tail_gates(Cols<D, HQ, HD> &r, const Who<D> &w, int nrow)
{
#pragma unroll
    for (int j = 0; j < r.N; ++j)
        if (item_row(w, j) >= nrow) r.g[j] = make_float2(0.f, 0.f);
}
// Gates (`in`, the next tile's or r.g itself) -> inclusive sums over the rows of the group in log2 units (r.g),
// the group's totals to sTot.
template <int D, bool HQ, bool HD>
__device__ __forceinline__ void group_prefix(Cols<D, HQ, HD> &r, const float2 (&in)[Cols<D, HQ, HD>::N], const Who<D> &w, float *sTot)
{
    const float2 l2e = make_float2(kLog2e, kLog2e);
    float2 run = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        run = fma2(in[j], l2e, run);
        r.g[j] = run;
    }
    *reinterpret_cast<float2 *>(sTot + w.grp * D + w.c2) = run;
    if constexpr (Col<D>::X) {
        float2 x = mul2(in[8], l2e);
#pragma unroll
        for (int k = 1; k < 8; k <<= 1) {
            const float px = __shfl_up_sync(0xffffffffu, x.x, 4 * k), py = __shfl_up_sync(0xffffffffu, x.y, 4 * k);
            if (w.xrow >= k) x = add2(x, make_float2(px, py));
        }
        r.g[8] = x;
        if (w.xrow == 7) *reinterpret_cast<float2 *>(sTot + w.grp * D + w.xc2) = x;
    }
}
// Sums of the group totals: over the groups before the thread's, and over all of them.  Identical in every
// warp of the CTA (same order of additions).
struct Tot {
    float2 before, all, xbefore, xall;
};
template <int D, bool WINDOW>
__device__ __forceinline__ Tot sum_totals(const float *sTot, const Who<D> &w, int w0, int w1)
{
    Tot t;
    t.before = t.all = t.xbefore = t.xall = make_float2(0.f, 0.f);
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        if (!WINDOW || (s >= w0 && s < w1)) {             // uniform over the warp
            if (s == w.grp) {
                t.before = t.all;
                t.xbefore = t.xall;
            }
            t.all = add2(t.all, *reinterpret_cast<const float2 *>(sTot + s * D + w.c2));
            if (Col<D>::X) t.xall = add2(t.xall, *reinterpret_cast<const float2 *>(sTot + s * D + w.xc2));
        }
    }
    return t;
}
template <int D> __device__ __forceinline__ Tot tile_totals(const float *sTot, const Who<D> &w) { return sum_totals<D, false>(sTot, w, 0, 8); }
// The same over the row groups [w0, w1) of one sub-chunk.  Out of line: tiles are seldom divided.
template <int D> __device__ __noinline__ Tot window_totals(const float *sTot, Who<D> w, int w0, int w1) { return sum_totals<D, true>(sTot, w, w0, w1); }
template <int D> __device__ __forceinline__ bool beyond(const Tot &t)        // uniform over the CTA
{
    const bool b = fmaxf(fabsf(t.all.x), fabsf(t.all.y)) > kSubLimit || (Col<D>::X && fmaxf(fabsf(t.xall.x), fabsf(t.xall.y)) > kSubLimit);
    return __any_sync(0xffffffffu, b) != 0;
}
// Sums over one half of the tile's groups (HALF = 0, 1).
template <int D, int HALF>
__device__ __forceinline__ Tot half_totals(const float *sTot, const Who<D> &w)
{
    Tot t;
    t.before = t.all = t.xbefore = t.xall = make_float2(0.f, 0.f);
#pragma unroll
    for (int s = 4 * HALF; s < 4 * HALF + 4; ++s) {
        if (s == w.grp) {
            t.before = t.all;
            t.xbefore = t.xall;
        }
        t.all = add2(t.all, *reinterpret_cast<const float2 *>(sTot + s * D + w.c2));
        if (Col<D>::X) t.xall = add2(t.xall, *reinterpret_cast<const float2 *>(sTot + s * D + w.xc2));
    }
    return t;
}
// Longest sub-chunk length (a power of two between kMinSub and `start`) for which every aligned window of
// the tile keeps |sum of gates| <= kSubLimit in every channel; kMinSub if none does (then the range bit of
// *status is set).  Uniform over the CTA.
template <int D>
__device__ __noinline__ int choose_window(const float *sTot, Who<D> w, int start, int *status)
{
    for (int s = start;; s >>= 1) {
        bool viol = false;
        for (int w0 = 0; w0 < 8; w0 += s / 8) {
            const Tot t = sum_totals<D, true>(sTot, w, w0, w0 + s / 8);
            viol |= beyond<D>(t);
        }
        if (!viol) return s;
        if (s <= kMinSub) {
            if (threadIdx.x == 0) atomicOr(status, kStatusRange);
            return s;
        }
    }
}
// How a kernel works a tile of two sub-chunks of 32 rows, with the same bits: not looked for (a pass each where the search finds
// them), looked for first and a pass each, or both in one pass.
enum Halves { kNoHalves, kHalvesApart, kHalvesTogether };
// Sub-chunk length of a tile whose totals are tt; tt becomes the totals of the (sub-)chunk the thread's rows are in.  Halves,
// which chunks of 32 ask for and which suffice for most tiles beyond the limit, are tried with sums over fixed groups (the
// search takes a few hundred cycles).
template <int D, bool HALVES>
__device__ __forceinline__ int divide_below(const float *sTot, const Who<D> &w, int sub_max, int *status, Tot &tt)
{
    if (HALVES && sub_max >= T / 2) {
        const Tot lo = half_totals<D, 0>(sTot, w), hi = half_totals<D, 1>(sTot, w);
        if (!beyond<D>(lo) && !beyond<D>(hi)) {
            tt = w.grp < 4 ? lo : hi;
            return T / 2;
        }
    }
    const int s = choose_window<D>(sTot, w, min(sub_max, HALVES ? T / 4 : T / 2), status), w0 = 8 * w.grp / s * (s / 8);
    tt = window_totals<D>(sTot, w, w0, w0 + s / 8);
    return s;
}
struct Divided {
    Tot tt;
    int s;
};
template <int D>
__device__ __noinline__ Divided divide_away(const float *sTot, Who<D> w, int sub_max, int *status)
{
    Divided d;
    d.s = divide_below<D, true>(sTot, w, sub_max, status, d.tt);
    return d;
}
// AWAY: in a function of its own, out of the way of launches that wait for their instructions.
template <int D, Halves HALVES, bool AWAY = false>
__device__ __forceinline__ int divide_tile(const float *sTot, const Who<D> &w, int sub_max, int *status, Tot &tt)
{
    if (sub_max >= T && !beyond<D>(tt)) return T;
    if (!AWAY) return divide_below<D, HALVES != kNoHalves>(sTot, w, sub_max, status, tt);
    const Divided d = divide_away<D>(sTot, w, sub_max, status);
    tt = d.tt;
    return d.s;
}

__device__ __forceinline__ void st_pair(char *tile, int o, float2 a) { *reinterpret_cast<uint32_t *>(tile + o) = pack_h2(a.x, a.y); }
__device__ __forceinline__ void st_zero(char *tile, int o) { *reinterpret_cast<uint32_t *>(tile + o) = 0u; }
template <int D> __device__ __forceinline__ int pair_offset(int row, int c2) { return (c2 >> 3) * Cfg<D>::CHT + 2 * (c2 & 7) + 16 * row; }
// tile offset of item j
template <int D> __device__ __forceinline__ int item_offset(const Who<D> &w, int j)
{
    return j < 8 ? pair_offset<D>(8 * w.grp, w.c2) + 16 * j : pair_offset<D>(8 * w.grp + w.xrow, w.xc2);
}

// Operand tiles from the thread's rows, r.g[j] = x the exponent (log2) of item j:
//   tK <- k 2^-x, tV <- v;  tQ <- q 2^x, tG <- dO.  `on` = false (uniform over the warp) writes zeros.
template <int D, bool HQ, bool HD>
__device__ __forceinline__ void build_rows(const Cols<D, HQ, HD> &r, const Who<D> &w, char *tQ, char *tK, char *tV, char *tG, bool on)
{
    if (on) {
#pragma unroll
        for (int j = 0; j < r.N; ++j) {
            const int o = item_offset(w, j);
            st_pair(tK, o, mul2(bf2(r.k[j]), ex2_neg2(r.g[j])));
            st_pair(tV, o, bf2(r.v[j]));
            if (HQ) st_pair(tQ, o, mul2(bf2(r.q[j]), ex2_2(r.g[j])));
            if (HD) st_pair(tG, o, bf2(r.d[j]));
        }
    } else {
#pragma unroll
        for (int j = 0; j < r.N; ++j) {
            const int o = item_offset(w, j);
            st_zero(tK, o);
            st_zero(tV, o);
            if (HQ) st_zero(tQ, o);
            if (HD) st_zero(tG, o);
        }
    }
}
// Row sums of the gates -> exponents (log2) of the items' decay factors.  Rows past the end of the sequence get 0: their
// operands are zero, and where the gates are beyond the range 2^x would overflow there and make them 0 * inf.
template <int D, bool HQ, bool HD>
__device__ __forceinline__ void centre_rows(Cols<D, HQ, HD> &r, const Who<D> &w, float2 off, float2 xoff, int nrow)
{
#pragma unroll
    for (int j = 0; j < r.N; ++j) r.g[j] = add2(r.g[j], j < 8 ? off : xoff);
    if (nrow < T) clear_tail_gates(r, w, nrow);
}
// exponent offset of a (sub-)chunk's rows: minus half its total, plus the groups before
__device__ __forceinline__ float2 centred(float2 before, float2 all) { return fma2(all, make_float2(-0.5f, -0.5f), before); }

// Sums of the group totals after the thread's group (in .before / .xbefore) and over all groups.
template <int D>
__device__ __forceinline__ Tot later_totals(const float *sTot, const Who<D> &w)
{
    Tot t;
    t.before = t.all = t.xbefore = t.xall = make_float2(0.f, 0.f);
#pragma unroll
    for (int s = 7; s >= 0; --s) {
        if (s == w.grp) {
            t.before = t.all;
            t.xbefore = t.xall;
        }
        t.all = add2(t.all, *reinterpret_cast<const float2 *>(sTot + s * D + w.c2));
        if (Col<D>::X) t.xall = add2(t.xall, *reinterpret_cast<const float2 *>(sTot + s * D + w.xc2));
    }
    return t;
}
// Where the backward sweep starts loading the next tile's rows: at d = 64 right after the operand tiles are
// built, at d = 72 (12 registers of state and rows more) after the accumulators have been read.
template <int D> constexpr bool kRowsEarly = D == 64;
// d = 72: the zero chunk behind the channels of tV, tG and tD and the zero rows of tD, which the accumulator buffers overwrite.
template <int D>
__device__ __forceinline__ void clear_pads(char *tV, char *tG, char *tD)
{
    using C = Cfg<D>;
    const uint4 z = make_uint4(0, 0, 0, 0);
    const int i = threadIdx.x;
    if (i < T) *reinterpret_cast<uint4 *>(tV + C::NCH * C::CHT + 16 * i) = z;
    else if (i < 2 * T) *reinterpret_cast<uint4 *>(tG + C::NCH * C::CHT + 16 * (i - T)) = z;
    else if (i < 2 * T + C::RS) *reinterpret_cast<uint4 *>(tD + C::NCH * C::CHS + 16 * (i - 2 * T)) = z;
    if (i < C::NCH * (C::RS - D)) {
        const int ch = i / (C::RS - D), r = D + i - ch * (C::RS - D);
        *reinterpret_cast<uint4 *>(tD + ch * C::CHS + 16 * r) = z;
    }
}

// ---- results through shared memory -------------------------------------------------------------------
// An accumulator row belongs to one lane, so a direct store (16 or 32 bytes per lane) touches 32 lines per
// instruction.  Rows go to a staging buffer instead and leave by the column threads, whole lines at a time:
// forward sweep with fp32 results 21.3 -> 15.5 us, backward 100 -> 94 us (48 sequences of 4096 tokens, d = 64; bf16
// results of the forward sweep: no difference).  The row stride is an odd number of 16-byte words (no bank conflicts).
template <int D, typename TO>
struct Staging {
    static constexpr int kStride = (D * (int)sizeof(TO) / 16 | 1) * 16;
    static constexpr int kBytes = T * kStride;
};
__device__ __forceinline__ void stage8(char *p, const float (&f)[8], float) { st8(reinterpret_cast<float *>(p), f); }
__device__ __forceinline__ void stage8(char *p, const float (&f)[8], bf16) { store_out8(reinterpret_cast<bf16 *>(p), f); }
// chunk jc of row `row`
template <int D, typename TO>
__device__ __forceinline__ void stage_row(char *stage, int row, int jc, const float (&f)[8])
{
    stage8(stage + row * Staging<D, TO>::kStride + 8 * jc * (int)sizeof(TO), f, TO());
}
template <typename TO> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<bf16> { using type = uint32_t; };
__device__ __forceinline__ void put_pair(float *dst, float2 v, bool add)
{
    if (add) asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" :: "l"(dst), "f"(v.x), "f"(v.y) : "memory");
    else *reinterpret_cast<float2 *>(dst) = v;
}
__device__ __forceinline__ void put_pair(bf16 *dst, uint32_t v, bool) { *reinterpret_cast<uint32_t *>(dst) = v; }
// The thread's items of the staged tile to global memory (rows below nrow), `oo` elements behind dst.  All shared-memory loads first: a
// load and a store per row in turn took 850 cycles per tile.
template <int D, typename TO>
__device__ __forceinline__ void flush_rows(TO *dst, uint32_t oo, const char *stage, const int *row_off, const Who<D> &w, int nrow, bool add)
{
    constexpr int N = Col<D>::X ? 9 : 8;
    uint32_t off[9];
    row_offsets<D>(row_off, w, off);
    typename Pair<TO>::type v[N];
#pragma unroll
    for (int j = 0; j < N; ++j)
        v[j] = *reinterpret_cast<const typename Pair<TO>::type *>(stage + item_row(w, j) * Staging<D, TO>::kStride + (j < 8 ? w.c2 : w.xc2) * (int)sizeof(TO));
    if (nrow == T) {
#pragma unroll
        for (int j = 0; j < N; ++j) put_pair(dst + (off[j] + oo), v[j], add);
    } else {
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (item_row(w, j) < nrow) put_pair(dst + (off[j] + oo), v[j], add);
    }
}

// ---- state of the recurrence (fp32 registers) ------------------------------------------------------
// Piece i of a thread: 8 value channels of key channel `row` (M = 64 product split by value chunks), or,
// at d = 72 on the warps cg = 1, i = 2, the transposed corner: value channel `xe`, key channels 64 .. 71.
template <int D>
struct StateOf {
    using C = Cfg<D>;
    using L = Col<D>;
    int row, cg, hf, xe;
    bool xok;
    __device__ __forceinline__ explicit StateOf(const Who<D> &w)
    {
        row = w.r16;
        cg = w.cg;
        hf = w.hf;
        xe = w.hf ? 64 + (w.r16 & 15) : w.r16;
        xok = w.hf == 0 || w.r16 < D - 64;
    }
    __device__ __forceinline__ bool corner(int i) const { return L::X && i == L::NPS - 1 && cg == 1; }       // uniform over the warp
    __device__ __forceinline__ int idx(int i) const { return cg + 2 * i; }
    __device__ __forceinline__ bool has(int i) const { return corner(i) || idx(i) < L::NV0; }         // uniform over the warp
    __device__ __forceinline__ bool mine(int i) const { return corner(i) ? xok : idx(i) < (hf ? L::NV1 : L::NV0); }
    __device__ __forceinline__ int chunk(int i) const { return (hf ? L::NV0 : 0) + idx(i); }
    __device__ __forceinline__ uint32_t tcol(int i) const { return corner(i) ? (uint32_t)L::HW : 8u * (uint32_t)idx(i); }
};
// Values per channel (the thread's own pairs, which every warp holds for all channels) -> the value of the thread's
// state row, and of key channel 64 + lane % 8 of the corner.
template <int D>
__device__ __forceinline__ float of_row(const StateOf<D> &st, float2 x)
{
    const float a = __shfl_sync(0xffffffffu, x.x, st.row >> 1), b = __shfl_sync(0xffffffffu, x.y, st.row >> 1);
    return (st.row & 1) ? b : a;
}
__device__ __forceinline__ float of_corner(float2 xx)
{
    const float a = __shfl_sync(0xffffffffu, xx.x, (threadIdx.x & 7) >> 1), b = __shfl_sync(0xffffffffu, xx.y, (threadIdx.x & 7) >> 1);
    return (threadIdx.x & 1) ? b : a;
}
// Gates (log2) summed over one (sub-)chunk or more, for the thread's state row and its corner channel.
struct RowSum {
    float t, xt;
};
template <int D>
__device__ __forceinline__ RowSum row_sum(const StateOf<D> &st, const Tot &tt)
{
    return RowSum{of_row(st, tt.all), Col<D>::X ? of_corner(tt.xall) : 0.f};
}
__device__ __forceinline__ RowSum operator+(RowSum a, RowSum b) { return RowSum{a.t + b.t, a.xt + b.xt}; }
// Decay of one (sub-)chunk whose gates sum to t: ec = 2^(t/2), e2c = 2^t for the thread's state row, x* for its corner channel.
struct Decay {
    float ec, e2c, xec, xe2c;
};
template <int D>
__device__ __forceinline__ Decay decay_of(RowSum r)
{
    Decay d;
    d.ec = ex2(0.5f * r.t);
    d.e2c = ex2(r.t);
    d.xec = Col<D>::X ? ex2(0.5f * r.xt) : 0.f;
    d.xe2c = Col<D>::X ? ex2(r.xt) : 0.f;
    return d;
}
// Weight of a (sub-)chunk's product in a sum over the segment: 2^x with x the decay from the chunk's centre to the
// segment's end (or from its start): half of the chunk's own gates `r` and those between, `far`.
struct Weight {
    float f, xf;
};
template <int D>
__device__ __forceinline__ Weight weight_of(RowSum r, RowSum far)
{
    return Weight{ex2(fmaf(0.5f, r.t, far.t)), Col<D>::X ? ex2(fmaf(0.5f, r.xt, far.xt)) : 0.f};
}
// the threads' row sums as an array over the channels (once per CTA)
template <int D>
__device__ __forceinline__ void put_row_sums(float *dst, const Who<D> &w, const StateOf<D> &st, RowSum r)
{
    if (w.cg == 0 && w.hf == 0) dst[st.row] = r.t;
    if (Col<D>::X && threadIdx.x < 8) dst[64 + threadIdx.x] = r.xt;
}
// value of key channel 64 + j of the corner (every lane of the warp must call it)
__device__ __forceinline__ float corner_val(float v, int j) { return __shfl_sync(0xffffffffu, v, j); }

// fp16 tile (row stride 16 B inside a chunk, chunk stride CH) <- diag(ec) S
template <int D, int CH>
__device__ __forceinline__ void put_state(char *tile, const StateOf<D> &m, const float (&S)[Col<D>::NPS][8], const Decay &d)
{
    using L = Col<D>;
#pragma unroll
    for (int i = 0; i < L::NPS; ++i) {
        if (!m.has(i)) continue;
        float x[8];
        if (m.corner(i)) {
            // rows are key channels, 16 bytes apart inside a value chunk
            char *p = tile + (m.xe >> 3) * CH + 64 * 16 + 2 * (m.xe & 7);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float f = corner_val(d.xec, e);
                x[e] = S[i][e] * f;
            }
            if (m.xok) {
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    const uint32_t h = pack_h2(x[e], x[e + 1]);
                    *reinterpret_cast<uint16_t *>(p + 16 * e) = (uint16_t)h;
                    *reinterpret_cast<uint16_t *>(p + 16 * e + 16) = (uint16_t)(h >> 16);
                }
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; e += 2) {
                const float2 y = mul2(make_float2(S[i][e], S[i][e + 1]), make_float2(d.ec, d.ec));
                x[e] = y.x;
                x[e + 1] = y.y;
            }
            if (m.mine(i)) *reinterpret_cast<uint4 *>(tile + m.chunk(i) * CH + m.row * 16) = pack_h8(x);
        }
    }
}
// S <- e2c S + ec U, U the accumulator at `acc`
template <int D>
__device__ __forceinline__ void fold_state(uint32_t acc, const StateOf<D> &m, float (&S)[Col<D>::NPS][8], const Decay &d)
{
    using L = Col<D>;
#pragma unroll
    for (int i = 0; i < L::NPS; ++i) {
        if (!m.has(i)) continue;
        float u[8];
        tmem_ld8(acc + m.tcol(i), u);
        if (m.corner(i)) {
#pragma unroll
            for (int e = 0; e < 8; ++e) S[i][e] = corner_val(d.xe2c, e) * S[i][e] + corner_val(d.xec, e) * u[e];
        } else {
#pragma unroll
            for (int e = 0; e < 8; e += 2) {
                const float2 x = fma2(make_float2(d.e2c, d.e2c), make_float2(S[i][e], S[i][e + 1]), mul2(make_float2(d.ec, d.ec), make_float2(u[e], u[e + 1])));
                S[i][e] = x.x;
                S[i][e + 1] = x.y;
            }
        }
    }
}
// sum <- sum + 2^x U, U the accumulator at `acc`, the sum in tensor memory too (`first`: nothing is there yet)
template <int D>
__device__ __forceinline__ void add_product(uint32_t sum, uint32_t acc, const StateOf<D> &m, const Weight &wt, bool first)
{
#pragma unroll
    for (int i = 0; i < Col<D>::NPS; ++i) {
        if (!m.has(i)) continue;
        float u[8], s[8];
        tmem_ld8_pair(acc + m.tcol(i), sum + m.tcol(i), u, s);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float f = m.corner(i) ? corner_val(wt.xf, e) : wt.f;
            s[e] = first ? f * u[e] : fmaf(f, u[e], s[e]);
        }
        tmem_st8(sum + m.tcol(i), s);
    }
    tmem_st_wait();
}
template <int D>
__device__ __forceinline__ void get_state(const float *src, const StateOf<D> &m, float (&S)[Col<D>::NPS][8])
{
#pragma unroll
    for (int i = 0; i < Col<D>::NPS; ++i) {
#pragma unroll
        for (int e = 0; e < 8; ++e) S[i][e] = 0.f;
        if (src && m.has(i) && m.mine(i)) {
            if (m.corner(i)) {
#pragma unroll
                for (int e = 0; e < 8; ++e) S[i][e] = src[(size_t)(64 + e) * D + m.xe];
            } else {
                ld8(src + (size_t)m.row * D + 8 * m.chunk(i), S[i]);
            }
        }
    }
}
template <int D>
__device__ __forceinline__ void save_state(float *dst, const StateOf<D> &m, const float (&S)[Col<D>::NPS][8])
{
#pragma unroll
    for (int i = 0; i < Col<D>::NPS; ++i)
        if (m.has(i) && m.mine(i)) {
            if (m.corner(i)) {
#pragma unroll
                for (int e = 0; e < 8; ++e) dst[(size_t)(64 + e) * D + m.xe] = S[i][e];
            } else {
                st8(dst + (size_t)m.row * D + 8 * m.chunk(i), S[i]);
            }
        }
}

// a state accumulator to a row-major [d][d] array
template <int D>
__device__ __forceinline__ void acc_to_global(uint32_t acc, const StateOf<D> &m, float *dst)
{
#pragma unroll
    for (int i = 0; i < Col<D>::NPS; ++i) {
        if (!m.has(i)) continue;
        float u[8];
        tmem_ld8(acc + m.tcol(i), u);
        if (!m.mine(i)) continue;
        if (m.corner(i)) {
#pragma unroll
            for (int e = 0; e < 8; ++e) dst[(size_t)(64 + e) * D + m.xe] = u[e];
        } else {
            st8(dst + (size_t)m.row * D + 8 * m.chunk(i), u);
        }
    }
}

// ---- products with split accumulators ----------------------------------------------------------------
constexpr uint32_t kHiLanes = 16u << 16;
// Rows a product takes: all of the tile, or one half where each half is a sub-chunk (the value is the quarters of the
// accumulator's lanes that hold the other rows).
enum Rows : uint32_t { kAllRows = 0, kLowRows = 0xc, kHighRows = 0x3 };
// acc <- A^T B over the token rows: rows = key channels (A), columns = value channels (B)
template <int D, Rows ROWS = kAllRows>
__device__ __forceinline__ void issue_state(uint32_t acc, const char *tA, const char *tB)
{
    using C = Cfg<D>;
    using L = Col<D>;
    constexpr int KS = ROWS == kAllRows ? T / 16 : T / 32;
    constexpr uint32_t first = ROWS == kHighRows ? T / 2 * 16 : 0;
    const uint32_t a = smem_u32(tA) + first, b = smem_u32(tB) + first;
    issue<64, 8 * L::NV0, true, true, KS, C::CHT, C::CHT>(acc, a, b, false);
    issue<64, 8 * L::NV1, true, true, KS, C::CHT, C::CHT>(acc + kHiLanes, a, b + L::NV0 * C::CHT, false);
    if (L::X) {
        // the corner, transposed: rows = value channels (64 and the remaining 8), columns = key channels 64 .. 71.
        // The second product's A operand covers chunks 8 .. 15, most of them beyond the tile: mapped shared
        // memory whose rows of the result nobody reads.
        issue<64, 8, true, true, KS, C::CHT, C::CHT>(acc + L::HW, b, a + 8 * C::CHT, false);
        issue<64, 8, true, true, KS, C::CHT, C::CHT>(acc + L::HW + kHiLanes, b + 8 * C::CHT, a + 8 * C::CHT, false);
    }
}
// acc (+)= A B with the value channels (columns of B) split; A K-major tile of 64 rows, B MN-major
template <int D, int KSTEPS, uint32_t BCH, Rows ROWS = kAllRows>
__device__ __forceinline__ void issue_split(uint32_t acc, const char *tA, const char *tB, bool accumulate)
{
    using C = Cfg<D>;
    using L = Col<D>;
    const uint32_t a = smem_u32(tA), b = smem_u32(tB);
    issue<64, 8 * L::NV0, false, true, KSTEPS, C::CHT, BCH, 128, ROWS>(acc, a, b, accumulate);
    issue<64, 8 * L::NV1, false, true, KSTEPS, C::CHT, BCH, 128, ROWS>(acc + kHiLanes, a, b + L::NV0 * BCH, accumulate);
}
// acc += P V, P the masked scores, the value channels split
template <int D>
__device__ __forceinline__ void issue_weighted(uint32_t acc, const char *tP, const char *tV)
{
    using C = Cfg<D>;
    using L = Col<D>;
    const uint32_t a = smem_u32(tP), b = smem_u32(tV);
    issue_triangle<8 * L::NV0, false, C::CHT, C::CHT>(acc, a, b);
    issue_triangle<8 * L::NV1, false, C::CHT, C::CHT>(acc + kHiLanes, a, b + L::NV0 * C::CHT);
}
// acc <- A B^T (scores), columns split into even (lanes 0-15) and odd (lanes 16-31) 8-token chunks
template <int D>
__device__ __forceinline__ void issue_scores(uint32_t acc, const char *tA, const char *tB)
{
    using C = Cfg<D>;
    const uint32_t a = smem_u32(tA), b = smem_u32(tB);
    issue<64, 32, false, false, C::KS, C::CHT, C::CHT, 256>(acc, a, b, false);
    issue<64, 32, false, false, C::KS, C::CHT, C::CHT, 256>(acc + kHiLanes, a, b + 128, false);
}

}  // namespace sw
}  // namespace dig
