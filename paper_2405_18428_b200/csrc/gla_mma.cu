// Warp-MMA kernel family for chunkwise gated linear attention (Eq. attn_gla, evaluated chunk by chunk
// as Section 3.5 describes): serves bf16 requests whose head sizes the tcgen05 family does not cover (any
// d_k, d_v that is a multiple of 8 up to 128, chunks of 16, 32, 64 or 128 tokens as far as shared memory
// allows) and the full gate.  Same decomposition
// as the other families: per-chunk state contributions, a scan over the chunks, then one CTA per
// (chunk, batch*head) for the outputs or the gradients.  Every contraction runs on the tensor cores
// through mma.sync.m16n8k8 (tf32 operands, fp32 accumulation) with fragments read straight from
// padded fp32 tiles in shared memory, so any multiple of 8 works as a contraction length and any
// multiple of 16 (after zero padding) as an output extent.  Operands are rounded to tf32 when the
// tiles are filled.  Requests in fp32 storage (served here only with the value-channel gate) keep full
// fp32 tiles instead and split every operand at fragment load into a tf32 head and a tf32 tail,
// x = hi + lo: three products hi*hi + lo*hi + hi*lo per fragment pair leave errors of order 2^-21,
// the accuracy fp32 storage is held to.
//
// What bounds it: the words of shared memory a fragment costs, and latency, since the fp32 tiles of a 64-token chunk leave
// room for one CTA of the gradient kernel per SM.  Hence all tiles of a kernel are loaded in one pass, the gradient
// kernel works in 32-row warp tiles, and products whose operands both lie along their rows spread over all banks.
// Full gate, 8 x 1024 tokens of 6 heads, d = C = 64 (us, before -> now): state 24 -> 20.4, with gradients 39 -> 30,
// outputs 35.6 -> 33.4, gradients 108 -> 88, and 13.5 for the value gate's sums over later chunks -> none (the gradient
// kernel takes them from the state leaving its chunk).
//
// Notation per chunk (rows j = 0..C-1 in scan order, zero rows past the end of the sequence):
//   Lam_j = inclusive prefix sum of the gates, gamma = exp(Lam_{C-1}),
//   Qt = q*exp(Lam), Kt = k*exp(-Lam), Kh = k*exp(Lam_{C-1}-Lam),
//   S = state entering the chunk, Dg = diag(gamma) * dL/d(state leaving the chunk); the scan kernels
//   leave both rounded to tf32 in the workspace.
#include <type_traits>

#include "dig_common.cuh"

namespace dig {
namespace {

using bf16 = __nv_bfloat16;
constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kMaxNB = 8;                    // 8-column fragments per warp tile: up to 64 columns

__host__ __device__ constexpr int pad16(int d) { return (d + 15) & ~15; }
// Row pitch (floats) of a tile whose rows hold `d` values: a multiple of 4 whose quarter is odd, so the
// 8 rows x 4 columns a fragment load touches fall into 32 different banks.
__host__ __device__ constexpr int pitch(int d) { return pad16(d) + 4; }
// The same for tiles whose padding columns are never read (every kernel but the state kernel, where d_k
// is an output extent and has to be a multiple of 16): d is a multiple of 8, so d / 4 + 1 is odd too.
__host__ __device__ constexpr int tight(int d) { return d + 4; }

// Sizes of a launch, either compile-time constants (the frequent shapes: strides fold into the
// instructions, loops unroll, divisions become shifts) or read from the geometry (everything else).
template <int C_, int DK_, int DV_>
struct FixedDims {
    static constexpr int kC = C_, kDK = DK_, kDV = DV_;      // 0 = not known at compile time
    __host__ __device__ explicit FixedDims(const Geom &) {}
    __device__ constexpr int C() const { return C_; }
    __device__ constexpr int dk() const { return DK_; }
    __device__ constexpr int dv() const { return DV_; }
};
struct AnyDims {
    static constexpr int kC = 0, kDK = 0, kDV = 0;
    int c_, dk_, dv_;
    __host__ __device__ explicit AnyDims(const Geom &g) : c_(g.C), dk_(g.dk), dv_(g.dv) {}
    __device__ int C() const { return c_; }
    __device__ int dk() const { return dk_; }
    __device__ int dv() const { return dv_; }
};

// Device-side arguments of the value-channel gate (unused by the kernels instantiated without it).
struct BetaDev {
    const float *bgate;     // log(beta) [B][L][H][d_v]
    float *gamma_v;         // [B*H][N][d_v]  exp of the chunk totals of bgate
    float *dbgate;          // gradient with respect to bgate (backward pass)
};

__device__ __forceinline__ float tf32r(float x)
{
    uint32_t u;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
    return __uint_as_float(u);
}

// Rounding of a tile element: none when the operands are split at fragment load (PR).
template <bool PR>
__device__ __forceinline__ float rnd(float x) { return PR ? x : tf32r(x); }
// x = hi + lo with hi the tf32 truncation of x (what the tensor core reads of an fp32 register anyway).
__device__ __forceinline__ void split_tf32(float x, uint32_t &hi, uint32_t &lo)
{
    hi = __float_as_uint(x) & 0xffffe000u;
    lo = __float_as_uint(x - __uint_as_float(hi));
}

__device__ __forceinline__ void mma8(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One warp: acc[mb][nb] += A(r0 + 16 mb .. + 15, k) * B(k, c0 + 8 nb .. + 7) for k in [k0, k1), mb < mbw, nb < nbw.
// A(m, k) = A[m*sam + k*sak], B(k, n) = Bm[k*sbk + n*sbn]; k0, k1 multiples of 8.
// Fragment layout of m16n8k8: with g = lane / 4, t = lane % 4 a lane holds A(g | g+8, t | t+4),
// B(t | t+4, g) and the results C(g | g+8, 2t | 2t+1).  The four + four lanes of a contraction step may hold any of its
// eight indices as long as A and B agree: where both operands lie with the contraction down their rows (strides
// sak = sbk = a row) they take 2t and 2t+1 (ALONG), which spreads rows a multiple of four words apart over all banks
// (t and t+4: two lanes to a bank).
template <bool PR, bool ALONG, int MB, int NB>
__device__ __forceinline__ void warp_mma(float (&acc)[MB][NB][4], const float *A, int sam, int sak, int r0,
                                         const float *Bm, int sbk, int sbn, int c0, int mbw, int nbw, int k0, int k1)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, t0 = ALONG ? 2 * t : t, dt = ALONG ? 1 : 4;
    const float *pa = A + (r0 + g) * sam + (t0 + k0) * sak;
    const float *pb = Bm + (t0 + k0) * sbk + (c0 + g) * sbn;
#pragma unroll 2
    for (int k = k0; k < k1; k += 8) {
        uint32_t a[MB][4], al[MB][4];
#pragma unroll
        for (int mb = 0; mb < MB; ++mb)
            if (mb < mbw) {
                const float *pm = pa + 16 * mb * sam;
                const float af[4] = {pm[0], pm[8 * sam], pm[dt * sak], pm[8 * sam + dt * sak]};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (PR) split_tf32(af[i], a[mb][i], al[mb][i]);
                    else a[mb][i] = __float_as_uint(af[i]);
                }
            }
#pragma unroll
        for (int nb = 0; nb < NB; ++nb)
            if (nb < nbw) {
                const float bf0 = pb[8 * nb * sbn], bf1 = pb[dt * sbk + 8 * nb * sbn];
                uint32_t b0 = __float_as_uint(bf0), b1 = __float_as_uint(bf1), b0l, b1l;
                if (PR) {
                    split_tf32(bf0, b0, b0l);
                    split_tf32(bf1, b1, b1l);
                }
#pragma unroll
                for (int mb = 0; mb < MB; ++mb)
                    if (mb < mbw) {
                        if (PR) {
                            mma8(acc[mb][nb], al[mb], b0, b1);          // the small terms first
                            mma8(acc[mb][nb], a[mb], b0l, b1l);
                        }
                        mma8(acc[mb][nb], a[mb], b0, b1);
                    }
            }
        pa += 8 * sak;
        pb += 8 * sbk;
    }
}
template <bool PR, bool ALONG, int NB>
__device__ __forceinline__ void warp_mma(float (&acc)[NB][4], const float *A, int sam, int sak, int r0,
                                         const float *Bm, int sbk, int sbn, int c0, int nbw, int k0, int k1)
{
    warp_mma<PR, ALONG>(reinterpret_cast<float (&)[1][NB][4]>(acc), A, sam, sak, r0, Bm, sbk, sbn, c0, 1, nbw, k0, k1);
}

template <int NB>
__device__ __forceinline__ void zero(float (&acc)[NB][4])
{
#pragma unroll
    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[nb][i] = 0.f;
}

// Calls f(row, col, v0, v1) for every pair of adjacent result columns this lane holds (col even).
template <int MB, int NB>
__device__ __forceinline__ void zero(float (&acc)[MB][NB][4])
{
#pragma unroll
    for (int mb = 0; mb < MB; ++mb) zero(acc[mb]);
}
template <int NB, typename F>
__device__ __forceinline__ void for_pairs(const float (&acc)[NB][4], int r0, int c0, int nbw, F f)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nb = 0; nb < NB; ++nb)
        if (nb < nbw) {
            f(r0 + g, c0 + 8 * nb + 2 * t, acc[nb][0], acc[nb][1]);
            f(r0 + g + 8, c0 + 8 * nb + 2 * t, acc[nb][2], acc[nb][3]);
        }
}

template <int MB, int NB, typename F>
__device__ __forceinline__ void for_pairs(const float (&acc)[MB][NB][4], int r0, int c0, int mbw, int nbw, F f)
{
#pragma unroll
    for (int mb = 0; mb < MB; ++mb)
        if (mb < mbw) for_pairs(acc[mb], r0 + 16 * mb, c0, nbw, f);
}

// The warp tiles of an M x N result (M a multiple of 16, N of 8): 16 rows by a group of 8-column
// fragments; the columns are split until every warp has a tile (the last group may be shorter).
__host__ __device__ constexpr int tile_splits(int M, int N)
{
    int cs = 1;
    while ((M >> 4) * cs < kWarps && cs < (N >> 3)) cs *= 2;
    return cs;
}
__host__ __device__ constexpr int tile_frags(int M, int N) { return ((N >> 3) + tile_splits(M, N) - 1) / tile_splits(M, N); }
// Fragments per warp tile as a compile-time bound: exact when both extents are known, else the maximum.
__host__ __device__ constexpr int frag_bound(int M, int N) { return (M > 0 && N > 0) ? tile_frags(M, N) : kMaxNB; }
// 8-column fragments of the gradient kernel's tiles of up to 32 rows: the columns are split until the tiles of one
// result are eight (two results side by side fill the warps), and to `most` fragments (registers: two accumulators each).
// 32 x 16 tiles read 16 words of shared memory a lane for four MMAs, 16 x 16 tiles 12 for two.
__host__ __device__ constexpr int grad_frags(int C, int N, int most)
{
    const int want = C >= 32 && C <= 256 ? 8 / ((C + 31) / 32) : 8, nf = N > 0 ? N >> 3 : 64;
    const int n = (nf + want - 1) / want;
    return C <= 0 || N <= 0 || n > most ? most : n;
}
struct Tiling {
    int nrt, nfrag, nbw, ntiles;
    __device__ Tiling(int M, int N) : nrt(M >> 4), nfrag(N >> 3), nbw(tile_frags(M, N)), ntiles((M >> 4) * tile_splits(M, N)) {}
    // first row, first column and fragment count (<= 0: nothing to do) of a tile
    __device__ void at(int tile, int &r0, int &c0, int &nbt) const
    {
        const int rt = tile % nrt, ct = tile / nrt;
        r0 = 16 * rt;
        c0 = 8 * nbw * ct;
        nbt = min(nbw, nfrag - nbw * ct);
    }
};

__device__ __forceinline__ float2 load2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ float2 load2(const __nv_bfloat16 *p) { return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p)); }
__device__ __forceinline__ void store2(float *p, float a, float b) { *reinterpret_cast<float2 *>(p) = make_float2(a, b); }
__device__ __forceinline__ void store2(__nv_bfloat16 *p, float a, float b)
{
    *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(a, b);
}

// ---- tile fills -----------------------------------------------------------------------------------
// sRow[j] = index of the chunk's row j among the (token, head) rows of a [B][L][H][.] tensor, or -1 past
// the end of the sequence.  Every later access to global memory goes through this table.
__device__ __forceinline__ void fill_rows(int *sRow, const Geom &g, int C, int b, int h, int chunk)
{
    for (int j = threadIdx.x; j < C; j += kThreads) {
        const int p = chunk * C + j;
        sRow[j] = p < g.L ? (b * g.L + scan_token(p, g.dir, g.gh, g.gw, g.L)) * g.H + h : -1;
    }
}
// Every tile is filled in one phase at the start of a kernel so that a CTA pays the latency of global
// memory once: fp32 sources travel by cp.async (no registers, all copies in flight together), bf16
// sources in register batches of four 8-byte loads per thread.  Rows past the end of the sequence and
// the padding columns become zero.  The values are rescaled / rounded in place afterwards.
__device__ __forceinline__ void cp_async16(float *dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}
// NT tiles with the same row length: all of a thread's loads of a pass are in flight together.
template <int NT>
__device__ __forceinline__ void load_tiles(float *const (&dst)[NT], int ld, const __nv_bfloat16 *const (&src)[NT], const int *sRow, int C, int d, int dp)
{
    constexpr int U = NT == 1 ? 4 : 2;
    const int per_row = dp >> 2, n = C * per_row;      // dp: columns to fill (d, or d padded to 16)
    for (int base = threadIdx.x; base < n; base += U * kThreads) {
        uint2 raw[U][NT];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = base + u * kThreads, j = idx / per_row, c = (idx - j * per_row) << 2;
            const int row = idx < n ? sRow[j] : -1;
#pragma unroll
            for (int i = 0; i < NT; ++i)
                raw[u][i] = row >= 0 && c < d ? *reinterpret_cast<const uint2 *>(src[i] + (size_t)row * d + c) : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = base + u * kThreads, j = idx / per_row, c = (idx - j * per_row) << 2;
            if (idx < n)
#pragma unroll
                for (int i = 0; i < NT; ++i)
                    *reinterpret_cast<float4 *>(dst[i] + j * ld + c) =
                        make_float4(lo_f(raw[u][i].x), hi_f(raw[u][i].x), lo_f(raw[u][i].y), hi_f(raw[u][i].y));
        }
    }
}
__device__ __forceinline__ void load_gates(float *dst, int ld, const float *gate, const int *sRow, int C, int dk, int dp)
{
    const int per_row = dp >> 2;
    for (int idx = threadIdx.x; idx < C * per_row; idx += kThreads) {
        const int j = idx / per_row, c = (idx - j * per_row) << 2;
        const int row = sRow[j];
        if (row >= 0 && c < dk) cp_async16(dst + j * ld + c, gate + (size_t)row * dk + c);
        else *reinterpret_cast<float4 *>(dst + j * ld + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}
template <int NT>
__device__ __forceinline__ void load_tiles(float *const (&dst)[NT], int ld, const float *const (&src)[NT], const int *sRow, int C, int d, int dp)
{
#pragma unroll
    for (int i = 0; i < NT; ++i) load_gates(dst[i], ld, src[i], sRow, C, d, dp);       // fp32 rows travel like the gates
}
// A [dk][dv] state of the workspace (rounded to tf32 by the scan kernels) -> [dk][ld] tile.
__device__ __forceinline__ void load_state(float *dst, int ld, const float *src, int dk, int dv)
{
    const int per_row = dv >> 2;
    for (int idx = threadIdx.x; idx < dk * per_row; idx += kThreads) {
        const int r = idx / per_row, c = (idx - r * per_row) << 2;
        if (r < dk && c < dv) cp_async16(dst + r * ld + c, src + r * dv + c);
        else *reinterpret_cast<float4 *>(dst + r * ld + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}
// First of the threads that work on the value-channel gate: behind those of the key-channel gate (four per channel)
// where the CTA has that many, else the same.
__device__ __forceinline__ int value_thread(int dkp, int dvp) { return 4 * (dkp + dvp) <= kThreads ? (int)threadIdx.x - 4 * dkp : (int)threadIdx.x; }

// In place: gates -> inclusive prefix sums down the rows of the chunk; sLast receives the last row.
// Four threads per channel take a quarter of the rows each; sSeg ([4][dkp]) carries the quarter totals.
// BETA: the same for the value-channel gate.  Contains two barriers.
template <bool BETA>
__device__ __forceinline__ void prefix_gates(float *lam, int ld, int C, int dkp, float *sLast, float *sSeg, float *lam_v, int ldv, int dvp, float *sLastV, float *sSegV)
{
    const int rows = C >> 2;                    // C is a multiple of 16
    auto sums = [&](float *x, int ldx, int dp, float *segs, int tid) -> float {
        const int c = tid % dp, seg = tid / dp;      // 4 * dp <= kThreads
        float run = 0.f;
        if (tid >= 0 && seg < 4) {
#pragma unroll 8
            for (int j = seg * rows; j < (seg + 1) * rows; ++j) {
                run += x[j * ldx + c];
                x[j * ldx + c] = run;
            }
            segs[seg * dp + c] = run;
        }
        return run;
    };
    auto shift = [&](float *x, int ldx, int dp, const float *segs, float *last, int tid, float run) {
        const int c = tid % dp, seg = tid / dp;
        if (tid >= 0 && seg < 4) {
            float add = 0.f;
            for (int sg = 0; sg < seg; ++sg) add += segs[sg * dp + c];
            if (seg > 0) {
#pragma unroll 8
                for (int j = seg * rows; j < (seg + 1) * rows; ++j) x[j * ldx + c] += add;
            }
            if (seg == 3) last[c] = run + add;
        }
    };
    const int tv = BETA ? value_thread(dkp, dvp) : 0;
    const float run = sums(lam, ld, dkp, sSeg, threadIdx.x), run_v = BETA ? sums(lam_v, ldv, dvp, sSegV, tv) : 0.f;
    __syncthreads();
    shift(lam, ld, dkp, sSeg, sLast, threadIdx.x, run);
    if (BETA) shift(lam_v, ldv, dvp, sSegV, sLastV, tv, run_v);
    __syncthreads();
}
// In place: sQ (raw q) -> Qt = q*exp(Lam), sK (raw k) -> Kt = k*exp(-Lam), or with sLast given
// -> Kh = k*exp(Lam_{C-1}-Lam); rounded to tf32.  Either tile may be null.
template <bool PR>
__device__ __forceinline__ void scale_qk(float *sQ, float *sK, const float *sLam, const float *sLast, int ldk, int C, int dp)
{
    const int per_row = dp >> 2;
    for (int idx = threadIdx.x; idx < C * per_row; idx += kThreads) {
        const int j = idx / per_row, c = (idx - j * per_row) << 2;
        const float4 lam = *reinterpret_cast<const float4 *>(sLam + j * ldk + c);
        if (sQ) {
            const float4 x = *reinterpret_cast<const float4 *>(sQ + j * ldk + c);
            *reinterpret_cast<float4 *>(sQ + j * ldk + c) = make_float4(
                rnd<PR>(x.x * __expf(lam.x)), rnd<PR>(x.y * __expf(lam.y)), rnd<PR>(x.z * __expf(lam.z)), rnd<PR>(x.w * __expf(lam.w)));
        }
        if (sK) {
            float4 e = make_float4(-lam.x, -lam.y, -lam.z, -lam.w);
            if (sLast) {
                const float4 last = *reinterpret_cast<const float4 *>(sLast + c);
                e = make_float4(last.x - lam.x, last.y - lam.y, last.z - lam.z, last.w - lam.w);
            }
            const float4 x = *reinterpret_cast<const float4 *>(sK + j * ldk + c);
            *reinterpret_cast<float4 *>(sK + j * ldk + c) = make_float4(
                rnd<PR>(x.x * __expf(e.x)), rnd<PR>(x.y * __expf(e.y)), rnd<PR>(x.z * __expf(e.z)), rnd<PR>(x.w * __expf(e.w)));
        }
    }
}

// sP[t][s] = A_t . B_s for s <= t, 0 above the diagonal, rounded to tf32 (A, B: [C][ld] tiles, contraction
// over the first K columns).  The diagonal has weight 1: the token's own k^T v enters undecayed.
template <int NB, bool PR>
__device__ __forceinline__ void masked_scores(float *sP, int ldp, const float *A, const float *Bm, int ld, int C, int K)
{
    const Tiling tl(C, C);
    const int warp = threadIdx.x >> 5;
    for (int tile = warp; tile < tl.ntiles; tile += kWarps) {
        int r0, c0, nbt;
        tl.at(tile, r0, c0, nbt);
        if (nbt <= 0) continue;
        float acc[NB][4];
        zero(acc);
        if (c0 <= r0 + 15) warp_mma<PR, false>(acc, A, ld, 1, r0, Bm, 1, ld, c0, nbt, 0, K);
        for_pairs(acc, r0, c0, nbt, [&](int t, int s, float v0, float v1) {
            *reinterpret_cast<float2 *>(sP + t * ldp + s) = make_float2(s <= t ? rnd<PR>(v0) : 0.f, s + 1 <= t ? rnd<PR>(v1) : 0.f);
        });
    }
}

// ---- kernel 1: chunk-local state contributions ------------------------------------------------------
// U = Kh^T V (and, for the backward pass, W = Qt^T dO); gamma = exp(Lam_{C-1}).
// BETA: with the value-channel gate the value side mirrors the key side: M = prefix sums of log(beta),
// gamma_v = exp(M_{C-1}), U = Kh^T Vh with Vh = v*exp(M_{C-1}-M), W = Qt^T G with G = dO*exp(M).
// CTAs per SM that the registers have to allow: with sizes not known at compile time two, which chunks that are short have the
// shared memory for (24 sequences of 6561 tokens, d = 48 x 88, chunks of 16 with the full gate: 493 us with 72 registers and one
// CTA, 312 with 64 and two); the others what their tiles allow.
template <typename DM> constexpr int kStateCtas = DM::kC == 0 ? 2 : DM::kC == 32 && DM::kDK == 64 ? 4 : 3;
template <bool BWD, typename DM, bool BETA, typename TI>
__global__ void __launch_bounds__(kThreads, kStateCtas<DM>)
mma_chunk_state(const TI *__restrict__ q, const TI *__restrict__ k, const TI *__restrict__ v, const float *__restrict__ gate,
                const TI *__restrict__ d_out, float *__restrict__ states, float *__restrict__ gamma,
                float *__restrict__ dstates, BetaDev bd, Geom g)
{
    constexpr bool PR = std::is_same<TI, float>::value;
    extern __shared__ __align__(16) float smem[];
    __shared__ int sRow[128];
    const DM dm(g);
    const int C = dm.C(), dk = dm.dk(), dv = dm.dv();
    const int chunk = blockIdx.x, bh = blockIdx.y, b = bh / g.H, h = bh - b * g.H;
    const int dkp = pad16(dk), dvp = pad16(dv), ldk = pitch(dk), ldv = pitch(dv);
    float *sLam = smem;                     // gates -> Lam
    float *sX = sLam + C * ldk;             // k -> Kh
    float *sV = sX + C * ldk;
    float *sLast = sV + C * ldv;            // [dkp]
    float *sSeg = sLast + dkp;              // [4][dkp]
    float *sQ = sSeg + 4 * dkp;             // BWD: q -> Qt
    float *sG = sQ + (BWD ? C * ldk : 0);   // BWD: dO
    float *sM = sG + (BWD ? C * ldv : 0);   // BETA: log(beta) -> M
    float *sMlast = sM + C * ldv;           // [dvp]
    float *sSegV = sMlast + dvp;            // [4][dvp]

    fill_rows(sRow, g, C, b, h, chunk);
    pdl_wait();
    pdl_launch_dependents();
    __syncthreads();
    if (BETA) load_gates(sM, ldv, bd.bgate, sRow, C, dv, dvp);
    load_gates(sLam, ldk, gate, sRow, C, dk, dkp);
    if (BWD && dk == dv) {
        load_tiles<4>({sX, sV, sQ, sG}, ldk, {k, v, q, d_out}, sRow, C, dk, dkp);
    } else if (BWD) {
        load_tiles<2>({sX, sQ}, ldk, {k, q}, sRow, C, dk, dkp);
        load_tiles<2>({sV, sG}, ldv, {v, d_out}, sRow, C, dv, dvp);
    } else if (dk == dv) {
        load_tiles<2>({sX, sV}, ldk, {k, v}, sRow, C, dk, dkp);
    } else {
        load_tiles<1>({sX}, ldk, {k}, sRow, C, dk, dkp);
        load_tiles<1>({sV}, ldv, {v}, sRow, C, dv, dvp);
    }
    cp_async_wait_all();
    __syncthreads();
    prefix_gates<BETA>(sLam, ldk, C, dkp, sLast, sSeg, sM, ldv, dvp, sMlast, sSegV);
    const size_t chunk_id = (size_t)bh * g.N + chunk;
    for (int c = threadIdx.x; c < dk; c += kThreads) gamma[chunk_id * dk + c] = __expf(sLast[c]);
    scale_qk<PR>(BWD ? sQ : nullptr, sX, sLam, sLast, ldk, C, dkp);
    if (BETA) {
        for (int e = threadIdx.x; e < dv; e += kThreads) bd.gamma_v[chunk_id * dv + e] = __expf(sMlast[e]);
        scale_qk<PR>(BWD ? sG : nullptr, sV, sM, sMlast, ldv, C, dvp);      // G = dO*exp(M), Vh = v*exp(M_{C-1}-M)
    }
    __syncthreads();
    constexpr int NB = frag_bound(pad16(DM::kDK), DM::kDV);
    const Tiling tl(dkp, dv);
    const int warp = threadIdx.x >> 5;
    float *U = states + chunk_id * dk * dv;
    float *W = BWD ? dstates + chunk_id * dk * dv : nullptr;
    for (int tile = warp; tile < tl.ntiles; tile += kWarps) {
        int r0, c0, nbt;
        tl.at(tile, r0, c0, nbt);
        if (nbt <= 0) continue;
        float acc[NB][4];
        zero(acc);
        warp_mma<PR, true>(acc, sX, 1, ldk, r0, sV, ldv, 1, c0, nbt, 0, C);           // sum_t Kh[t][c] V[t][e]
        for_pairs(acc, r0, c0, nbt, [&](int c, int e, float v0, float v1) {
            if (c < dk && e < dv) store2(U + c * dv + e, v0, v1);
        });
        if (BWD) {
            zero(acc);
            warp_mma<PR, true>(acc, sQ, 1, ldk, r0, sG, ldv, 1, c0, nbt, 0, C);       // sum_t Qt[t][c] dO[t][e]
            for_pairs(acc, r0, c0, nbt, [&](int c, int e, float v0, float v1) {
                if (c < dk && e < dv) store2(W + c * dv + e, v0, v1);
            });
        }
    }
}

// ---- kernel 3: outputs ------------------------------------------------------------------------------
// out = tril(Qt Kt^T) V + Qt S
// BETA: out = exp(M) * (tril(Qt Kt^T) Vt + Qt S) with Vt = v*exp(-M).
template <typename TO, typename DM, bool BETA, typename TI>
__global__ void __launch_bounds__(kThreads)
mma_chunk_out(const TI *__restrict__ q, const TI *__restrict__ k, const TI *__restrict__ v, const float *__restrict__ gate,
              const float *__restrict__ states, TO *__restrict__ out, BetaDev bd, Geom g)
{
    constexpr bool PR = std::is_same<TI, float>::value;
    extern __shared__ __align__(16) float smem[];
    __shared__ int sRow[128];
    const DM dm(g);
    const int C = dm.C(), dk = dm.dk(), dv = dm.dv();
    const int chunk = blockIdx.x, bh = blockIdx.y, b = bh / g.H, h = bh - b * g.H;
    const int dkp = dk, ldk = tight(dk), ldv = tight(dv), ldp = tight(C);      // no padding columns here
    float *sLam = smem;
    float *sQ = sLam + C * ldk;
    float *sK = sQ + C * ldk;
    float *sV = sK + C * ldk;
    float *sS = sV + C * ldv;               // [dkp][ldv]
    float *sLast = sS + dkp * ldv;          // [dkp]
    float *sSeg = sLast + dkp;              // [4][dkp]
    float *sP = (C <= dk) ? sLam : sSeg + 4 * dkp;       // the scores reuse the gate tile when they fit
    float *sM = sSeg + 4 * dkp + (C <= dk ? 0 : C * ldp);   // BETA: log(beta) -> M
    float *sMlast = sM + C * ldv;           // [dv]
    float *sSegV = sMlast + dv;             // [4][dv]

    fill_rows(sRow, g, C, b, h, chunk);
    __syncthreads();
    // the inputs of the call: whatever produced them has completed before the kernels in front of this one started
    if (BETA) load_gates(sM, ldv, bd.bgate, sRow, C, dv, dv);
    load_gates(sLam, ldk, gate, sRow, C, dk, dk);
    if (dk == dv) {
        load_tiles<3>({sV, sQ, sK}, ldk, {v, q, k}, sRow, C, dk, dk);
    } else {
        load_tiles<2>({sQ, sK}, ldk, {q, k}, sRow, C, dk, dk);
        load_tiles<1>({sV}, ldv, {v}, sRow, C, dv, dv);
    }
    pdl_wait();                             // the states come from the scan in front
    pdl_launch_dependents();
    load_state(sS, ldv, states + ((size_t)bh * g.N + chunk) * dk * dv, dk, dv);
    cp_async_wait_all();
    __syncthreads();
    prefix_gates<BETA>(sLam, ldk, C, dkp, sLast, sSeg, sM, ldv, dv, sMlast, sSegV);
    scale_qk<PR>(sQ, sK, sLam, nullptr, ldk, C, dk);
    if (BETA) scale_qk<PR>(nullptr, sV, sM, nullptr, ldv, C, dv);           // Vt = v*exp(-M)
    __syncthreads();
    masked_scores<frag_bound(DM::kC, DM::kC), PR>(sP, ldp, sQ, sK, ldk, C, dk);
    __syncthreads();
    constexpr int NB = frag_bound(DM::kC, DM::kDV);
    const Tiling tl(C, dv);
    const int warp = threadIdx.x >> 5;
    for (int tile = warp; tile < tl.ntiles; tile += kWarps) {
        int r0, c0, nbt;
        tl.at(tile, r0, c0, nbt);
        if (nbt <= 0) continue;
        float acc[NB][4];
        zero(acc);
        warp_mma<PR, false>(acc, sP, ldp, 1, r0, sV, ldv, 1, c0, nbt, 0, r0 + 16);     // columns past the diagonal are zero
        warp_mma<PR, false>(acc, sQ, ldk, 1, r0, sS, ldv, 1, c0, nbt, 0, dk);
        for_pairs(acc, r0, c0, nbt, [&](int j, int e, float v0, float v1) {
            const int row = sRow[j];
            if (BETA) {
                const float2 m = load2(sM + j * ldv + e);
                v0 *= __expf(m.x);
                v1 *= __expf(m.y);
            }
            if (row >= 0 && e < dv) store2(out + (size_t)row * dv + e, v0, v1);
        });
    }
}

// ---- kernel 4: gradients ----------------------------------------------------------------------------
//   P = tril(Qt Kt^T),  dP = tril(dO V^T)
//   dq = (dP Kt + dO S^T) * exp(Lam)
//   dk = (dP^T Qt + V Dg^T) * exp(-Lam)
//   dv = P^T dO + Kt Dg
//   dgate_j = carry + sum_{r >= j in chunk} (q*dq - k*dk)_r,   q*dq = Qt*(dq accumulator), k*dk alike
// BETA: the same formulas with Vt = v*exp(-M) for V and G = dO*exp(M) for dO (Dg then carries both
// decays); dv = (P^T G + Kt Dg) * exp(-M), and the gradient of log(beta) is, mirroring dgate,
//   dbgate_j = carry_v + sum_{r >= j in chunk} (o*dO - v*dv)_r  with  o*dO = (P Vt + Qt S)*G  and  v*dv = Vt*(dv accumulator)
// (the unscaled output P Vt + Qt S is recomputed here, two more products, rather than read back in
// storage precision).  carry_v, the sum over the later chunks, is sum_c S' D over the state leaving the chunk.
template <typename TO, typename DM, bool BETA, typename TI>
__global__ void __launch_bounds__(kThreads)
mma_chunk_bwd(const TI *__restrict__ q, const TI *__restrict__ k, const TI *__restrict__ v, const float *__restrict__ gate,
              const TI *__restrict__ d_out, const float *__restrict__ states,
              const float *__restrict__ dstates, const float *__restrict__ carry, TO *__restrict__ dq,
              TO *__restrict__ dk_out, TO *__restrict__ dv_out, float *__restrict__ dgate, BetaDev bd, Geom g)
{
    constexpr bool PR = std::is_same<TI, float>::value;
    extern __shared__ __align__(16) float smem[];
    __shared__ int sRow[128];
    const DM dm(g);
    const int C = dm.C(), dk = dm.dk(), dv = dm.dv();
    const int chunk = blockIdx.x, bh = blockIdx.y, b = bh / g.H, h = bh - b * g.H;
    const int dkp = dk, ldk = tight(dk), ldv = tight(dv), ldp = tight(C);      // no padding columns here
    float *sLam = smem;                     // Lam, later x = q*dq - k*dk
    float *sQ = sLam + C * ldk;
    float *sK = sQ + C * ldk;
    float *sV = sK + C * ldk;
    float *sG = sV + C * ldv;               // dO
    float *sS = sG + C * ldv;               // [dkp][ldv]
    float *sD = sS + dkp * ldv;             // [dkp][ldv]  Dg, as the scan kernel stores it
    float *sP = sD + dkp * ldv;             // [C][ldp]
    float *sdP = sP + C * ldp;              // [C][ldp]
    float *sLast = sdP + C * ldp;           // [dkp]
    float *sSeg = sLast + dkp;              // [4][dkp]
    float *sM = sSeg + 4 * dkp;             // BETA: log(beta) -> M, later x = o*dO - v*dv
    float *sMlast = sM + C * ldv;           // [dv]
    float *sSegV = sMlast + dv;             // [4][dv]
    const size_t chunk_id = (size_t)bh * g.N + chunk;

    fill_rows(sRow, g, C, b, h, chunk);
    __syncthreads();
    // the inputs of the call: whatever produced them has completed before the kernels in front of this one started
    if (BETA) load_gates(sM, ldv, bd.bgate, sRow, C, dv, dv);
    load_gates(sLam, ldk, gate, sRow, C, dk, dk);
    if (dk == dv) {
        load_tiles<4>({sV, sG, sQ, sK}, ldk, {v, d_out, q, k}, sRow, C, dk, dk);
    } else {
        load_tiles<2>({sQ, sK}, ldk, {q, k}, sRow, C, dk, dk);
        load_tiles<2>({sV, sG}, ldv, {v, d_out}, sRow, C, dv, dv);
    }
    pdl_wait();                             // the states come from the scans in front
    pdl_launch_dependents();
    load_state(sS, ldv, states + chunk_id * dk * dv, dk, dv);
    load_state(sD, ldv, dstates + chunk_id * dk * dv, dk, dv);
    cp_async_wait_all();
    __syncthreads();
    prefix_gates<BETA>(sLam, ldk, C, dkp, sLast, sSeg, sM, ldv, dv, sMlast, sSegV);
    scale_qk<PR>(sQ, sK, sLam, nullptr, ldk, C, dk);
    if (BETA) scale_qk<PR>(sG, sV, sM, nullptr, ldv, C, dv);                // G = dO*exp(M), Vt = v*exp(-M)
    __syncthreads();
    masked_scores<frag_bound(DM::kC, DM::kC), PR>(sP, ldp, sQ, sK, ldk, C, dk);
    masked_scores<frag_bound(DM::kC, DM::kC), PR>(sdP, ldp, sG, sV, ldv, C, dv);
    __syncthreads();
    // Warp tiles of up to 32 rows, first those of dv (BETA: and of the outputs), then those of dq and dk
    constexpr int MB = DM::kC == 16 ? 1 : 2, kMost = PR ? 2 : 4;
    constexpr int NBV = grad_frags(DM::kC, DM::kDV, kMost), NBK = grad_frags(DM::kC, DM::kDK, kMost);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gi = lane >> 2, ti = lane & 3;
    const int nrt = (C + 31) >> 5, nfv = grad_frags(C, dv, kMost), nfk = grad_frags(C, dk, kMost);
    const int ntv = nrt * (((dv >> 3) + nfv - 1) / nfv), ntk = nrt * (((dk >> 3) + nfk - 1) / nfk);
    const int mbw = C >= 32 ? 2 : 1;
    for (int tile = warp; tile < ntv + ntk; tile += kWarps) {
        if (tile < ntv) {
            // dv[s][e] = sum_c Kt[s][c] Dg[c][e] + sum_{t >= s} P[t][s] dO[t][e]
            const int rt = tile % nrt, ct = tile / nrt, r0 = 32 * rt, c0 = 8 * nfv * ct, nbt = min(nfv, (dv >> 3) - nfv * ct);
            float acc[MB][NBV][4];
            zero(acc);
            warp_mma<PR, false>(acc, sK, ldk, 1, r0, sD, ldv, 1, c0, mbw, nbt, 0, dk);
            if (BETA) {
                // column sums of Vt * (Kt Dg) over this tile's rows, part of what later chunks hand to dbgate
#pragma unroll
                for (int nb = 0; nb < NBV; ++nb)
                    if (nb < nbt) {
                        float2 sum = make_float2(0.f, 0.f);
#pragma unroll
                        for (int mb = 0; mb < MB; ++mb)
                            if (mb < mbw) {
#pragma unroll
                                for (int i = 0; i < 4; i += 2) {
                                    const float2 vt = load2(sV + (r0 + 16 * mb + gi + 4 * i) * ldv + c0 + 8 * nb + 2 * ti);
                                    sum.x = fmaf(vt.x, acc[mb][nb][i], sum.x);
                                    sum.y = fmaf(vt.y, acc[mb][nb][i + 1], sum.y);
                                }
                            }
#pragma unroll
                        for (int off = 4; off < 32; off <<= 1) {
                            sum.x += __shfl_xor_sync(0xffffffffu, sum.x, off);
                            sum.y += __shfl_xor_sync(0xffffffffu, sum.y, off);
                        }
                        if (gi == 0) *reinterpret_cast<float2 *>(sSegV + rt * dv + c0 + 8 * nb + 2 * ti) = sum;
                    }
            }
            warp_mma<PR, true>(acc, sP, 1, ldp, r0, sG, ldv, 1, c0, mbw, nbt, r0, C);
            if (BETA) {
                // unscaled output of the same tile, then x = o*dO - v*dv = (P Vt + Qt S)*G - Vt*(dv accumulator)
                float oh[MB][NBV][4];
                zero(oh);
                warp_mma<PR, false>(oh, sP, ldp, 1, r0, sV, ldv, 1, c0, mbw, nbt, 0, min(r0 + 32, C));
                warp_mma<PR, false>(oh, sQ, ldk, 1, r0, sS, ldv, 1, c0, mbw, nbt, 0, dk);
#pragma unroll
                for (int mb = 0; mb < MB; ++mb)
#pragma unroll
                    for (int nb = 0; nb < NBV; ++nb)
                        if (mb < mbw && nb < nbt) {
#pragma unroll
                            for (int i = 0; i < 4; i += 2) {
                                const int off = (r0 + 16 * mb + gi + 4 * i) * ldv + c0 + 8 * nb + 2 * ti;
                                const float2 vt = load2(sV + off), gg = load2(sG + off);
                                oh[mb][nb][i] = oh[mb][nb][i] * gg.x - vt.x * acc[mb][nb][i];
                                oh[mb][nb][i + 1] = oh[mb][nb][i + 1] * gg.y - vt.y * acc[mb][nb][i + 1];
                            }
                        }
                // this thread alone touches its elements of M: scale dv by exp(-M), then leave x there
                for_pairs(acc, r0, c0, mbw, nbt, [&](int j, int e, float v0, float v1) {
                    const int row = sRow[j];
                    const float2 m = load2(sM + j * ldv + e);
                    if (row >= 0) store2(dv_out + (size_t)row * dv + e, v0 * __expf(-m.x), v1 * __expf(-m.y));
                });
                __syncwarp();
                for_pairs(oh, r0, c0, mbw, nbt, [&](int j, int e, float v0, float v1) {
                    *reinterpret_cast<float2 *>(sM + j * ldv + e) = make_float2(v0, v1);
                });
            } else {
                for_pairs(acc, r0, c0, mbw, nbt, [&](int j, int e, float v0, float v1) {
                    const int row = sRow[j];
                    if (row >= 0) store2(dv_out + (size_t)row * dv + e, v0, v1);
                });
            }
        } else {
            // dq and dk of the same (row, channel) tile; x = q*dq - k*dk replaces Lam, element by element
            const int tk = tile - ntv, rt = tk % nrt, ct = tk / nrt, r0 = 32 * rt, c0 = 8 * nfk * ct, nbt = min(nfk, (dk >> 3) - nfk * ct);
            float acc[MB][NBK][4], xq[MB][NBK][4];
            auto times = [&](const float *t, auto f) {       // f(x, t * accumulator) for every result of this lane
#pragma unroll
                for (int mb = 0; mb < MB; ++mb)
#pragma unroll
                    for (int nb = 0; nb < NBK; ++nb)
                        if (mb < mbw && nb < nbt) {
#pragma unroll
                            for (int i = 0; i < 4; i += 2) {
                                const float2 tt = load2(t + (r0 + 16 * mb + gi + 4 * i) * ldk + c0 + 8 * nb + 2 * ti);
                                f(xq[mb][nb][i], tt.x * acc[mb][nb][i]);
                                f(xq[mb][nb][i + 1], tt.y * acc[mb][nb][i + 1]);
                            }
                        }
            };
            zero(acc);
            warp_mma<PR, false>(acc, sdP, ldp, 1, r0, sK, ldk, 1, c0, mbw, nbt, 0, min(r0 + 32, C));      // sum_{s <= t} dP[t][s] Kt[s][c]
            warp_mma<PR, false>(acc, sG, ldv, 1, r0, sS, 1, ldv, c0, mbw, nbt, 0, dv);                    // sum_e dO[t][e] S[c][e]
            times(sQ, [](float &x, float y) { x = y; });
            for_pairs(acc, r0, c0, mbw, nbt, [&](int j, int c, float v0, float v1) {
                const int row = sRow[j];
                const float2 lam = load2(sLam + j * ldk + c);
                if (row >= 0) store2(dq + (size_t)row * dk + c, v0 * __expf(lam.x), v1 * __expf(lam.y));
            });
            zero(acc);
            warp_mma<PR, true>(acc, sdP, 1, ldp, r0, sQ, ldk, 1, c0, mbw, nbt, r0, C);                    // sum_{t >= s} dP[t][s] Qt[t][c]
            warp_mma<PR, false>(acc, sV, ldv, 1, r0, sD, 1, ldv, c0, mbw, nbt, 0, dv);                    // sum_e V[s][e] Dg[c][e]
            times(sK, [](float &x, float y) { x -= y; });
            for_pairs(acc, r0, c0, mbw, nbt, [&](int j, int c, float v0, float v1) {
                const int row = sRow[j];
                const float2 lam = load2(sLam + j * ldk + c);
                if (row >= 0) store2(dk_out + (size_t)row * dk + c, v0 * __expf(-lam.x), v1 * __expf(-lam.y));
            });
            __syncwarp();
            for_pairs(xq, r0, c0, mbw, nbt, [&](int j, int c, float v0, float v1) {
                *reinterpret_cast<float2 *>(sLam + j * ldk + c) = make_float2(v0, v1);
            });
        }
    }
    __syncthreads();
    // gate gradients: suffix sums of x down the chunk plus what later chunks carry in; four threads per
    // channel take a quarter of the rows each
    {
        const int rows = C >> 2;
        const int c = threadIdx.x % dkp, seg = threadIdx.x / dkp;
        const float from_later = seg < 4 ? carry[chunk_id * dk + c] : 0.f;
        float run = 0.f;
        if (seg < 4) {
#pragma unroll 8
            for (int j = (seg + 1) * rows - 1; j >= seg * rows; --j) {
                run += sLam[j * ldk + c];
                sLam[j * ldk + c] = run;
            }
            sSeg[seg * dkp + c] = run;
        }
        // The value-channel gate: the same.  Later chunks hand over sum_c S'[c][e] D[c][e] with S' the state leaving
        // the chunk, = sum_c S Dg + sum_s Vt (Kt Dg)[s][e]: a quarter of the first sum and the rows that the warps above
        // left in sSegV per thread, exchanged through the spent score tiles.
        const int tv = BETA ? value_thread(dkp, dv) : -1, cv = tv % dv, segv = tv / dv;
        const bool on_v = tv >= 0 && segv < 4;
        if (BETA && on_v) {
            float part = segv < nrt ? sSegV[segv * dv + cv] : 0.f;
#pragma unroll 8
            for (int r = segv * dk / 4; r < (segv + 1) * dk / 4; ++r) part = fmaf(sS[r * ldv + cv], sD[r * ldv + cv], part);
            sP[segv * dv + cv] = part;
            float runv = 0.f;
#pragma unroll 8
            for (int j = (segv + 1) * rows - 1; j >= segv * rows; --j) {
                runv += sM[j * ldv + cv];
                sM[j * ldv + cv] = runv;
            }
            sSegV[segv * dv + cv] = runv;
        }
        __syncthreads();
        if (seg < 4) {
            float add = from_later;
            for (int sg = seg + 1; sg < 4; ++sg) add += sSeg[sg * dkp + c];
#pragma unroll 8
            for (int j = seg * rows; j < (seg + 1) * rows; ++j) {
                const int row = sRow[j];
                const float x = sLam[j * ldk + c] + add;
                if (row >= 0) dgate[(size_t)row * dk + c] = x;
            }
        }
        if (BETA && on_v) {
            float add = sP[cv] + sP[dv + cv] + sP[2 * dv + cv] + sP[3 * dv + cv];
            for (int sg = segv + 1; sg < 4; ++sg) add += sSegV[sg * dv + cv];
#pragma unroll 8
            for (int j = segv * rows; j < (segv + 1) * rows; ++j) {
                const int row = sRow[j];
                const float x = sM[j * ldv + cv] + add;
                if (row >= 0) bd.dbgate[(size_t)row * dv + cv] = x;
            }
        }
    }
}

size_t smem_state(const Geom &g, bool bwd, bool beta)
{
    size_t n = (size_t)g.C * (pitch(g.dk) * (bwd ? 3 : 2) + pitch(g.dv) * (bwd ? 2 : 1)) + 5 * pad16(g.dk);
    if (beta) n += (size_t)g.C * pitch(g.dv) + 5 * pad16(g.dv);
    return sizeof(float) * n;
}
size_t smem_out(const Geom &g, bool beta)
{
    size_t n = (size_t)g.C * (3 * tight(g.dk) + tight(g.dv)) + (size_t)g.dk * tight(g.dv) + 5 * g.dk;
    if (g.C > g.dk) n += (size_t)g.C * tight(g.C);
    if (beta) n += (size_t)g.C * tight(g.dv) + 5 * g.dv;
    return sizeof(float) * n;
}
size_t smem_bwd(const Geom &g, bool beta)
{
    size_t n = (size_t)g.C * (3 * tight(g.dk) + 2 * tight(g.dv) + 2 * tight(g.C)) + 2 * (size_t)g.dk * tight(g.dv) + 5 * g.dk;
    if (beta) n += (size_t)g.C * tight(g.dv) + 5 * g.dv;
    return sizeof(float) * n;
}
constexpr size_t kMaxSmem = 227 * 1024 - 1024;      // the row table is static shared memory

template <typename K>
dig_status set_smem(K kernel, size_t bytes)
{
    if (bytes > kMaxSmem) return DIG_ERR_UNSUPPORTED;
    return ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), bytes);
}

// The value-channel gate keeps one more block behind the common workspace: gamma_v [B*H][N][d_v].
size_t beta_block(const Geom &g) { return align256((size_t)g.B * g.H * g.N * g.dv * sizeof(float)); }
BetaDev beta_dev(const GlaArgs &a, const Workspace &w, bool backward)
{
    BetaDev bd{};
    if (a.bio.bgate == nullptr) return bd;
    char *p = reinterpret_cast<char *>(a.ws) + w.bytes;
    bd.bgate = a.bio.bgate;
    bd.gamma_v = reinterpret_cast<float *>(p);
    if (backward) bd.dbgate = a.bio.dbgate;
    return bd;
}

template <typename TO, typename DM, bool BETA, typename TI = bf16>
dig_status fwd_dims(const GlaArgs &a)
{
    constexpr bool kRound = !std::is_same<TI, float>::value;     // states rounded to tf32 by the scans
    const Geom &g = a.g;
    const Workspace w = carve_workspace(a.ws, g, false);
    const BetaDev bd = beta_dev(a, w, false);
    const dim3 grid(g.N, g.B * g.H);
    dig_status st;
    auto k1 = mma_chunk_state<false, DM, BETA, TI>;
    if ((st = set_smem(k1, smem_state(g, false, BETA))) != DIG_OK) return st;
    auto k3 = mma_chunk_out<TO, DM, BETA, TI>;
    if ((st = set_smem(k3, smem_out(g, BETA))) != DIG_OK) return st;
    {
        KernelTimer t(KID_MMA_STATE, a.stream);
        launch_pdl(k1, grid, dim3(kThreads), smem_state(g, false, BETA), a.stream, (const TI *)a.q, (const TI *)a.k, (const TI *)a.v,
                   a.gate, (const TI *)nullptr, w.states, w.gamma, (float *)nullptr, bd, g);
    }
    if (BETA) st = launch_state_scan_fwd_beta(w, bd.gamma_v, g, a.stream, kRound);
    else st = launch_state_scan_fwd(w, g, a.stream, a.sio, kRound);
    if (st != DIG_OK) return st;
    KernelTimer t(KID_MMA_OUT, a.stream);
    launch_pdl(k3, grid, dim3(kThreads), smem_out(g, BETA), a.stream, (const TI *)a.q, (const TI *)a.k, (const TI *)a.v, a.gate,
               (const float *)w.states, (TO *)a.out, bd, g);
    return cuda_ok(cudaGetLastError());
}

template <typename TO, typename DM, bool BETA, typename TI = bf16>
dig_status bwd_dims(const GlaArgs &a)
{
    constexpr bool kRound = !std::is_same<TI, float>::value;
    const Geom &g = a.g;
    const Workspace w = carve_workspace(a.ws, g, true);
    const BetaDev bd = beta_dev(a, w, true);
    const dim3 grid(g.N, g.B * g.H);
    dig_status st;
    auto k1 = mma_chunk_state<true, DM, BETA, TI>;
    if ((st = set_smem(k1, smem_state(g, true, BETA))) != DIG_OK) return st;
    auto k4 = mma_chunk_bwd<TO, DM, BETA, TI>;
    if ((st = set_smem(k4, smem_bwd(g, BETA))) != DIG_OK) return st;
    {
        KernelTimer t(KID_MMA_STATE, a.stream);
        launch_pdl(k1, grid, dim3(kThreads), smem_state(g, true, BETA), a.stream, (const TI *)a.q, (const TI *)a.k, (const TI *)a.v,
                   a.gate, (const TI *)a.d_out, w.states, w.gamma, w.dstates, bd, g);
    }
    if (BETA) {
        if ((st = launch_state_scan_fwd_beta(w, bd.gamma_v, g, a.stream, kRound)) != DIG_OK) return st;
        if ((st = launch_state_scan_bwd_beta(w, bd.gamma_v, g, a.stream, kRound)) != DIG_OK) return st;
    } else {
        if ((st = launch_state_scan_fwd(w, g, a.stream, a.sio, kRound)) != DIG_OK) return st;
        if ((st = launch_state_scan_bwd(w, g, a.stream, a.sio, kRound)) != DIG_OK) return st;
    }
    {
        KernelTimer t(KID_MMA_BWD, a.stream);
        launch_pdl(k4, grid, dim3(kThreads), smem_bwd(g, BETA), a.stream, (const TI *)a.q, (const TI *)a.k, (const TI *)a.v, a.gate,
                   (const TI *)a.d_out, (const float *)w.states, (const float *)w.dstates, (const float *)w.carry, (TO *)a.dq,
                   (TO *)a.dk, (TO *)a.dv, a.dgate, bd, g);
    }
    return cuda_ok(cudaGetLastError());
}

// Head sizes and chunks of the paper's models get kernels with compile-time sizes (6 heads of 64, 8 x 1024 tokens in
// chunks of 32 with the full gate: 546 -> 225 us; 4 x 1024 tokens in fp32: 249 -> 141).  Without the full gate these heads
// are the tcgen05 family's: the two instances kept there serve calls that force this family.
template <bool BETA, typename F>
dig_status with_dims(const Geom &g, F f)
{
    if (g.dk == 72 && g.dv == 72 && g.C == 64) return f(FixedDims<64, 72, 72>(g));
    if (g.dk == 64 && g.dv == 64 && g.C == 32) return f(FixedDims<32, 64, 64>(g));
    if constexpr (BETA) {
        if (g.dk == 64 && g.dv == 64 && g.C == 64) return f(FixedDims<64, 64, 64>(g));
        if (g.dk == 72 && g.dv == 72 && g.C == 32) return f(FixedDims<32, 72, 72>(g));
    }
    return f(AnyDims(g));
}
template <typename TO, bool BETA, typename TI = bf16>
dig_status fwd_typed(const GlaArgs &a)
{
    return with_dims<BETA>(a.g, [&](auto dm) { return fwd_dims<TO, decltype(dm), BETA, TI>(a); });
}
template <typename TO, bool BETA, typename TI = bf16>
dig_status bwd_typed(const GlaArgs &a)
{
    return with_dims<BETA>(a.g, [&](auto dm) { return bwd_dims<TO, decltype(dm), BETA, TI>(a); });
}

}  // namespace

bool mma_supports(int dk, int dv, int chunk, int dtype, bool backward, bool beta)
{
    if (dtype == DIG_F32 && !beta) return false;      // fp32 storage: only the full gate is served here (split operands)
    Geom g{};
    g.dk = dk; g.dv = dv; g.C = chunk;
    if (backward) return smem_bwd(g, beta) <= kMaxSmem && smem_state(g, true, beta) <= kMaxSmem;
    return smem_out(g, beta) <= kMaxSmem && smem_state(g, false, beta) <= kMaxSmem;
}

size_t mma_beta_workspace_bytes(const Geom &g, bool backward)
{
    return carve_workspace(nullptr, g, backward).bytes + beta_block(g);
}

dig_status mma_gla_fwd(const GlaArgs &a)
{
    const bool beta = a.bio.bgate != nullptr;
    if (a.dtype == DIG_BF16) return beta ? fwd_typed<__nv_bfloat16, true>(a) : fwd_typed<__nv_bfloat16, false>(a);
    if (a.dtype == DIG_BF16_F32OUT) return beta ? fwd_typed<float, true>(a) : fwd_typed<float, false>(a);
    if (a.dtype == DIG_F32 && beta) return fwd_typed<float, true, float>(a);
    return DIG_ERR_UNSUPPORTED;
}

dig_status mma_gla_bwd(const GlaArgs &a)
{
    const bool beta = a.bio.bgate != nullptr;
    if (a.dtype == DIG_BF16) return beta ? bwd_typed<__nv_bfloat16, true>(a) : bwd_typed<__nv_bfloat16, false>(a);
    if (a.dtype == DIG_BF16_F32OUT) return beta ? bwd_typed<float, true>(a) : bwd_typed<float, false>(a);
    if (a.dtype == DIG_F32 && beta) return bwd_typed<float, true, float>(a);
    return DIG_ERR_UNSUPPORTED;
}

}  // namespace dig
