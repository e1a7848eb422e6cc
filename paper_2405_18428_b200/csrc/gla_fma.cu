// fp32-FMA kernel family for chunkwise gated linear attention (Eq. attn_gla, evaluated chunk
// by chunk as Section 3.5 describes).  Serves DIG_F32 (products must be fp32-accurate, which a
// single tf32 tensor-core pass is not) and any bf16 request the tensor-core family does not
// cover.  One CTA per (chunk, batch*head), or several where few chunks leave SMs idle (share); every contraction is a
// register-blocked FMA loop over shared-memory tiles: 4x4 blocks in the state and output kernels, 8x4 in the gradient kernel.
//
// What bounds it: latency.  A CTA holds a whole chunk (C = d = 64 in fp32: 80 to 160 KB) and 192 chunks fill 148 SMs
// once or twice, so a kernel's time is one or two CTAs' serial chain of load, prefix, scores, products.  Hence all
// tiles of a kernel are asked for at once, prefix sums run in segments on all threads, loops are unrolled so that
// several shared loads are in flight, and rounds and waits in front of the states' arrival are filled by the
// programmatic launch.  B = 2, H = 6, L = 1024, d = C = 64 (us, before -> now): state 18 -> 11.2, with gradients
// 26 -> 16.9, outputs 29 -> 21.2, gradients 100 -> 58; one 256-token sequence of 6 heads, whose
// chunks are shared: state 14.7 -> 5.8, outputs 21.4 -> 12.4.
//
// Notation per chunk (rows j = 0..C-1 in scan order, zero rows past the end of the sequence):
//   Lam_j = inclusive prefix sum of the gates, gamma = exp(Lam_{C-1}),
//   Qt = q*exp(Lam), Kt = k*exp(-Lam), Kh = k*exp(Lam_{C-1}-Lam) = Kt*gamma,
//   S = state entering the chunk, D = dL/d(state leaving the chunk).
#include "dig_common.cuh"

namespace dig {
namespace {

constexpr int kThreads = 256;        // state and output kernels
constexpr int kBwdThreads = 512;     // gradient kernel, at most
// Threads of the gradient kernel: 128 registers each fill an SM with one CTA of a 64-token chunk or two of a shorter one
__host__ __device__ inline int bwd_threads(int C) { return C >= 64 ? kBwdThreads : kBwdThreads / 2; }

// ---- 4x4 register-blocked contractions over shared memory --------------------------------
// acc[i][j] += sum_k A[(r0+i)*lda + k] * Bm[(c0 + j*cstep)*ldb + k], columns j < jn only (jn uniform enough over a
// warp to skip whole pieces of a causal product)
__device__ __forceinline__ void mm_nt(float (&acc)[4][4], const float *A, int lda, int r0,
                                      const float *Bm, int ldb, int c0, int cstep, int K, int jn)
{
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float4 a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4 *>(A + (r0 + i) * lda + k);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < jn) {
                const float4 b = *reinterpret_cast<const float4 *>(Bm + (c0 + j * cstep) * ldb + k);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    acc[i][j] += a[i].x * b.x + a[i].y * b.y + a[i].z * b.z + a[i].w * b.w;
            }
    }
}
// acc[i][j] += sum_{k<K} A[(r0+i)*lda + k] * Bm[k*ldb + c0 + j]
template <int UNROLL>
__device__ __forceinline__ void mm_nn(float (&acc)[4][4], const float *A, int lda, int r0,
                                      const float *Bm, int ldb, int c0, int K)
{
#pragma unroll UNROLL
    for (int k = 0; k < K; k += 4) {
        float4 a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4 *>(A + (r0 + i) * lda + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) b[kk] = *reinterpret_cast<const float4 *>(Bm + (k + kk) * ldb + c0);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc[i][0] += a[i].x * b[0].x + a[i].y * b[1].x + a[i].z * b[2].x + a[i].w * b[3].x;
            acc[i][1] += a[i].x * b[0].y + a[i].y * b[1].y + a[i].z * b[2].y + a[i].w * b[3].y;
            acc[i][2] += a[i].x * b[0].z + a[i].y * b[1].z + a[i].z * b[2].z + a[i].w * b[3].z;
            acc[i][3] += a[i].x * b[0].w + a[i].y * b[1].w + a[i].z * b[2].w + a[i].w * b[3].w;
        }
    }
}
// acc[i][j] += sum_{k<K} A[k*lda + r0 + i] * Bm[k*ldb + c0 + j]
__device__ __forceinline__ void mm_tn(float (&acc)[4][4], const float *A, int lda, int r0,
                                      const float *Bm, int ldb, int c0, int K)
{
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
        const float4 a = *reinterpret_cast<const float4 *>(A + k * lda + r0);
        const float4 b = *reinterpret_cast<const float4 *>(Bm + k * ldb + c0);
        const float av[4] = {a.x, a.y, a.z, a.w};
        const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] += av[i] * bv[j];
    }
}
__device__ __forceinline__ void zero(float (&acc)[4][4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
}

// ---- 8x4 blocks of the gradient kernel -------------------------------------------------------------
// Eight rows from r0, four columns cb, cb + cs, cb + 2 cs, cb + 3 cs: neighbouring lanes read neighbouring rows
// (nt: an odd number of 16-byte words apart) or columns of B, so no access conflicts, and 12 loads feed 128
// multiply-adds (4x4 blocks on neighbouring columns: 8 feed 64, and the nt products hit two banks eight times).
struct Acc8 {
    float v[8][4];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) v[i][j] = 0.f;
    }
};
// += sum_k A[(r0+i)*lda + k] * B[(cb + j*cs)*ldb + k]
__device__ __forceinline__ void mm8_nt(Acc8 &acc, const float *A, int lda, int r0, const float *B, int ldb, int cb, int cs, int K)
{
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float4 b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4 *>(B + (cb + j * cs) * ldb + k);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 a = *reinterpret_cast<const float4 *>(A + (r0 + i) * lda + k);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc.v[i][j] += a.x * b[j].x + a.y * b[j].y + a.z * b[j].z + a.w * b[j].w;
        }
    }
}
// += sum_{k<K} A[(r0+i)*lda + k] * scale[k] * B[k*ldb + cb + j*cs]   (SCALED: with the factor)
template <bool SCALED>
__device__ __forceinline__ void mm8_nn(Acc8 &acc, const float *A, int lda, int r0, const float *B, int ldb, int cb, int cs, int K, const float *scale)
{
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float b[4][4];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int j = 0; j < 4; ++j) b[kk][j] = B[(k + kk) * ldb + cb + j * cs];
        float4 sc = make_float4(1.f, 1.f, 1.f, 1.f);
        if (SCALED) sc = *reinterpret_cast<const float4 *>(scale + k);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float4 a = *reinterpret_cast<const float4 *>(A + (r0 + i) * lda + k);
            if (SCALED) a = make_float4(a.x * sc.x, a.y * sc.y, a.z * sc.z, a.w * sc.w);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc.v[i][j] += a.x * b[0][j] + a.y * b[1][j] + a.z * b[2][j] + a.w * b[3][j];
        }
    }
}
// += sum_{k0<=k<K} A[k*lda + r0 + i] * B[k*ldb + cb + j*cs]
__device__ __forceinline__ void mm8_tn(Acc8 &acc, const float *A, int lda, int r0, const float *B, int ldb, int cb, int cs, int k0, int K)
{
#pragma unroll 4
    for (int k = k0; k < K; ++k) {
        const float4 a0 = *reinterpret_cast<const float4 *>(A + k * lda + r0), a1 = *reinterpret_cast<const float4 *>(A + k * lda + r0 + 4);
        const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float b = B[k * ldb + cb + j * cs];
#pragma unroll
            for (int i = 0; i < 8; ++i) acc.v[i][j] = fmaf(a[i], b, acc.v[i][j]);
        }
    }
}

// ---- tile loaders ----------------------------------------------------------------------------
// Row table: (token, head) row of the chunk's row j in a [B][L][H][.] tensor, -1 past the end of the sequence.  It
// lies in the padding behind the rows of a tile.
struct Rows {
    int *p;
    int ld;
    __device__ __forceinline__ Rows(float *tile, int ld_, int d) : p(reinterpret_cast<int *>(tile + d)), ld(ld_) {}
    __device__ __forceinline__ int operator[](int j) const { return p[j * ld]; }
};
__device__ __forceinline__ void fill_rows(const Rows &rows, const Geom &g, int b, int h, int chunk)
{
    for (int j = threadIdx.x; j < g.C; j += blockDim.x) {
        const int p = chunk * g.C + j;
        rows.p[j * rows.ld] = p < g.L ? (b * g.L + scan_token(p, g.dir, g.gh, g.gw, g.L)) * g.H + h : -1;
    }
}
// Copies the chunk's rows of a [B][L][H][d] tensor into shared memory (row stride ld floats), rows past the end
// of the sequence become zero.  fp32 travels by cp.async, so that all tiles of a kernel are in flight together and
// a CTA pays the latency of global memory once; loads_done() before the barrier that publishes them.
__device__ __forceinline__ void cp_async16(float *dst, const float *src, bool on)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void loads_done() { asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory"); }
// Rows j0 .. j1 - 1 (kept at their places), `w` of the d columns from src on.
__device__ __forceinline__ void load_tile(float *dst, int ld, const float *src, const Rows &sRow, int j0, int j1, int d, int w)
{
    const int per_row = w >> 2, n = (j1 - j0) * per_row;
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        const int r = idx / per_row, j = j0 + r, c = (idx - r * per_row) << 2, row = sRow[j];
        cp_async16(dst + j * ld + c, src + (size_t)max(row, 0) * d + c, row >= 0);
    }
}
__device__ __forceinline__ void load_tile(float *dst, int ld, const __nv_bfloat16 *src, const Rows &sRow, int j0, int j1, int d, int w)
{
    const int per_row = w >> 2, n = (j1 - j0) * per_row;
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        const int r = idx / per_row, j = j0 + r, c = (idx - r * per_row) << 2, row = sRow[j];
        *reinterpret_cast<float4 *>(dst + j * ld + c) = row >= 0 ? load4(src + (size_t)row * d + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}
template <typename T>
__device__ __forceinline__ void load_tile(float *dst, int ld, const T *src, const Rows &sRow, int C, int d) { load_tile(dst, ld, src, sRow, 0, C, d, d); }
// A [dk][dv] state of the workspace -> [dk][ld] tile.
__device__ __forceinline__ void load_state(float *dst, int ld, const float *src, int dk, int dv)
{
    const int per_row = dv >> 2, n = dk * per_row;
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        const int r = idx / per_row, c = (idx - r * per_row) << 2;
        cp_async16(dst + r * ld + c, src + 4 * (size_t)idx, true);
    }
}

// In place: gates -> inclusive prefix sums down the rows; the rows are cut in as many segments as there are
// threads per channel, whose totals go through sSeg ([segments][dk] floats).  Contains two barriers, the last at the end.
__device__ __forceinline__ void prefix_gates(float *lam, int ld, int C, int dk, float *sSeg)
{
    const int nseg = min((int)blockDim.x / dk, 8), rows = (C + nseg - 1) / nseg;
    const int seg = threadIdx.x / dk, c = threadIdx.x - seg * dk, j0 = seg * rows, j1 = min(j0 + rows, C);
    if (seg < nseg) {
        float run = 0.f;
#pragma unroll 8
        for (int j = j0; j < j1; ++j) {
            run += lam[j * ld + c];
            lam[j * ld + c] = run;
        }
        sSeg[seg * dk + c] = run;
    }
    __syncthreads();
    if (seg < nseg && seg > 0) {
        float add = 0.f;
        for (int s = 0; s < seg; ++s) add += sSeg[s * dk + c];
#pragma unroll 8
        for (int j = j0; j < j1; ++j) lam[j * ld + c] += add;
    }
    __syncthreads();
}
__device__ __forceinline__ float4 exp4(float4 x) { return make_float4(expf(x.x), expf(x.y), expf(x.z), expf(x.w)); }
__device__ __forceinline__ float4 mul4(float4 a, float4 b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }

// ---- kernel 1: chunk-local state contributions ------------------------------------------------
// U = Kh^T V  (and, for the backward pass, W = Qt^T dO); gamma = exp(Lam_{C-1}).  CTA z of a chunk takes a slice of the key
// channels (SHARED: where the chunks leave SMs idle).
template <typename T, bool BWD, bool SHARED>
__global__ void __launch_bounds__(kThreads)
fma_chunk_state(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v,
                const float *__restrict__ gate, const T *__restrict__ d_out,
                float *__restrict__ states, float *__restrict__ gamma, float *__restrict__ dstates,
                Geom g)
{
    extern __shared__ __align__(16) float smem[];
    const int chunk = blockIdx.x, bh = blockIdx.y, b = bh / g.H, h = bh - b * g.H;
    const int w = SHARED ? g.dk / gridDim.z : g.dk, k0 = SHARED ? blockIdx.z * w : 0;      // the CTA's key channels
    const int ldk = w + 4, ldv = g.dv + 4;
    float *sLam = smem;                     // gates -> Lam
    float *sX = sLam + g.C * ldk;           // k -> Kh
    float *sV = sX + g.C * ldk;
    float *sSeg = sV + g.C * ldv;           // [8][w]
    float *sQ = sSeg + 8 * w;               // BWD: Qt
    float *sG = sQ + (BWD ? g.C * ldk : 0); // BWD: dO

    const Rows sRow(sV, ldv, g.dv);
    fill_rows(sRow, g, b, h, chunk);
    pdl_wait();
    pdl_launch_dependents();
    __syncthreads();
    load_tile(sLam, ldk, gate + k0, sRow, 0, g.C, g.dk, w);
    load_tile(sX, ldk, k + k0, sRow, 0, g.C, g.dk, w);
    load_tile(sV, ldv, v, sRow, g.C, g.dv);
    if (BWD) {
        load_tile(sQ, ldk, q + k0, sRow, 0, g.C, g.dk, w);
        load_tile(sG, ldv, d_out, sRow, g.C, g.dv);
    }
    loads_done();
    __syncthreads();
    prefix_gates(sLam, ldk, g.C, w, sSeg);
    const size_t chunk_id = (size_t)bh * g.N + chunk;
    const float *sLast = sLam + (g.C - 1) * ldk;
    for (int c = threadIdx.x; c < w; c += kThreads) gamma[chunk_id * g.dk + k0 + c] = expf(sLast[c]);
    {
        const int per_row = w >> 2;
        for (int idx = threadIdx.x; idx < g.C * per_row; idx += kThreads) {
            const int j = idx / per_row, o = j * ldk + ((idx - j * per_row) << 2);
            const float4 lam = *reinterpret_cast<const float4 *>(sLam + o), last = *reinterpret_cast<const float4 *>(sLast + o - j * ldk);
            const float4 e = exp4(make_float4(last.x - lam.x, last.y - lam.y, last.z - lam.z, last.w - lam.w));
            *reinterpret_cast<float4 *>(sX + o) = mul4(*reinterpret_cast<const float4 *>(sX + o), e);
            if (BWD) *reinterpret_cast<float4 *>(sQ + o) = mul4(*reinterpret_cast<const float4 *>(sQ + o), exp4(lam));
        }
    }
    __syncthreads();
    const int nrb = w >> 2, ncb = g.dv >> 2;
    float *U = states + (chunk_id * g.dk + k0) * g.dv;
    float *W = BWD ? dstates + (chunk_id * g.dk + k0) * g.dv : nullptr;
    for (int blk = threadIdx.x; blk < nrb * ncb; blk += kThreads) {
        const int r0 = (blk / ncb) << 2, c0 = (blk % ncb) << 2;
        float acc[4][4];
        zero(acc);
        mm_tn(acc, sX, ldk, r0, sV, ldv, c0, g.C);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4 *>(U + (r0 + i) * g.dv + c0) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        if (BWD) {
            zero(acc);
            mm_tn(acc, sQ, ldk, r0, sG, ldv, c0, g.C);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                *reinterpret_cast<float4 *>(W + (r0 + i) * g.dv + c0) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        }
    }
}

// In place: q -> Qt = q exp(Lam), k -> Kt = k exp(-Lam), Lam -> exp(Lam); q from row q0 on.
__device__ __forceinline__ void make_qt_kt(float *sQ, float *sK, float *sLam, int ldk, int C, int dk, int q0 = 0)
{
    const int per_row = dk >> 2;
    for (int idx = threadIdx.x; idx < C * per_row; idx += blockDim.x) {
        const int j = idx / per_row, o = j * ldk + ((idx - j * per_row) << 2);
        const float4 lam = *reinterpret_cast<const float4 *>(sLam + o), e = exp4(lam);
        *reinterpret_cast<float4 *>(sLam + o) = e;
        if (j >= q0) *reinterpret_cast<float4 *>(sQ + o) = mul4(*reinterpret_cast<const float4 *>(sQ + o), e);
        *reinterpret_cast<float4 *>(sK + o) = mul4(*reinterpret_cast<const float4 *>(sK + o), exp4(make_float4(-lam.x, -lam.y, -lam.z, -lam.w)));
    }
}

// One 4x4 block (rows r0.., columns cb, cb+nb, ..) of P[t][s] = A_t . B_s for s <= t, 0 above the diagonal (the
// token's own k^T v enters undecayed, so the diagonal weight is exactly q_t . k_t).
__device__ __forceinline__ void score_block(float *sP, int ldp, const float *sA, int lda, const float *sB, int ldb, int C, int K, int blk)
{
    const int nb = C >> 2, r0 = (blk / nb) << 2, cb = blk % nb;
    float acc[4][4];
    zero(acc);
    mm_nt(acc, sA, lda, r0, sB, ldb, cb, nb, K, (r0 + 3) / nb + 1);       // columns from j * nb > r0 + 3 on lie above the diagonal
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int s = cb + j * nb;
            sP[(r0 + i) * ldp + s] = (s <= r0 + i) ? acc[i][j] : 0.f;
        }
}

// ---- kernel 3: outputs ---------------------------------------------------------------------------
// out = tril(Qt Kt^T) V + Qt S
// CTA z of a chunk takes a part of its rows, for which it needs the keys up to them (SHARED: where the chunks leave SMs
// idle; parts are whole quarters, so that the interleaved columns of a score block stay below the part's last row).
// PERSM: CTAs per SM that the registers allow, three, or four on shorter loops where a launch has more CTAs than three per SM and
// shared memory holds four (chunks below 64): 180 sequences of 250 tokens in chunks of 16 (d = 64) take 82 us with three, 70
// with four.  Fewer CTAs are faster with three (12 sequences of 1024 tokens in chunks of 32: 31.0 us a pass, 34.7 with four).
template <typename T, typename TO, int PERSM, bool SHARED>
__global__ void __launch_bounds__(kThreads, PERSM)
fma_chunk_out(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v,
              const float *__restrict__ gate, const float *__restrict__ states,
              TO *__restrict__ out, Geom g)
{
    extern __shared__ __align__(16) float smem[];
    const int chunk = blockIdx.x, bh = blockIdx.y, b = bh / g.H, h = bh - b * g.H;
    const int ldk = g.dk + 4, ldv = g.dv + 4, ldp = g.C + 4;
    const int rows = SHARED ? g.C / gridDim.z : g.C, lo = SHARED ? blockIdx.z * rows : 0, hi = lo + rows;     // the CTA's rows; keys below hi
    float *sLam = smem;
    float *sQ = sLam + g.C * ldk;
    float *sK = sQ + g.C * ldk;
    float *sV = sK + g.C * ldk;
    float *sS = sV + g.C * ldv;             // [dk][ldv]
    float *sSeg = sS;                       // [8][dk], before the state arrives
    float *sP = sLam;                       // scores reuse the gate buffer once Qt, Kt exist
    // (sP needs C*(C+4) <= C*(dk+4) floats only when C <= dk; otherwise it gets its own space)
    if (g.C > g.dk) sP = sS + g.dk * ldv;

    const Rows sRow(sV, ldv, g.dv);
    fill_rows(sRow, g, b, h, chunk);
    __syncthreads();
    // the inputs of the call: whatever produced them has completed before the kernels in front of this one started
    load_tile(sLam, ldk, gate, sRow, hi, g.dk);
    load_tile(sV, ldv, v, sRow, hi, g.dv);
    load_tile(sQ, ldk, q, sRow, lo, hi, g.dk, g.dk);
    load_tile(sK, ldk, k, sRow, hi, g.dk);
    loads_done();
    __syncthreads();
    prefix_gates(sLam, ldk, hi, g.dk, sSeg);
    make_qt_kt(sQ, sK, sLam, ldk, hi, g.dk, lo);
    __syncthreads();
    pdl_wait();                             // the states come from the scan in front
    pdl_launch_dependents();
    load_state(sS, ldv, states + ((size_t)bh * g.N + chunk) * g.dk * g.dv, g.dk, g.dv);
    const int nb = g.C >> 2;
    for (int blk = (lo >> 2) * nb + threadIdx.x; blk < (hi >> 2) * nb; blk += kThreads) score_block(sP, ldp, sQ, ldk, sK, ldk, g.C, g.dk, blk);
    loads_done();
    __syncthreads();
    constexpr int UN = PERSM > 3 ? 1 : 4;
    const int nrb = rows >> 2, ncb = g.dv >> 2;
    for (int blk = threadIdx.x; blk < nrb * ncb; blk += kThreads) {
        const int r0 = lo + ((blk / ncb) << 2), c0 = (blk % ncb) << 2;
        float acc[4][4];
        zero(acc);
        mm_nn<UN>(acc, sP, ldp, r0, sV, ldv, c0, r0 + 4);       // columns beyond the diagonal are zero
        mm_nn<UN>(acc, sQ, ldk, r0, sS, ldv, c0, g.dk);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = sRow[r0 + i];
            if (row >= 0) store4(out + (size_t)row * g.dv + c0, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
        }
    }
}

// ---- kernel 4: gradients ---------------------------------------------------------------------------
//   dP = tril(dO V^T)
//   dq = (dP Kt + dO S^T) * exp(Lam)
//   dk = (dP^T Qt) * exp(-Lam) + (V D^T) * exp(Lam_{C-1}-Lam)
//   dv = P^T dO + Kh D
//   dgate_j = carry + sum_{r >= j in chunk} (q*dq - k*dk)_r
// After the scores, three groups of whole warps compute the blocks of dq, dk and dv side by side in registers: one
// CTA of 512 threads per SM, 128 registers each (256 threads with 4x4 blocks took 87 us where this takes 58).  With
// s = dP^T Qt + gamma (V D^T), dk = s / exp(Lam), q*dq = Qt (dq accumulator) and k*dk = Kt s.
__host__ __device__ inline int grad_blocks(int C, int d) { return ((C / 8) * (d / 4) + 31) & ~31; }
// The tile of q*dq - k*dk lies over the score tiles where it fits and one round of blocks is all there is.
__host__ __device__ inline bool x_over_scores(int C, int dk, int dv)
{
    return dk + 4 <= 2 * (C + 4) && 2 * grad_blocks(C, dk) + grad_blocks(C, dv) <= bwd_threads(C);
}
template <typename T, typename TO>
__global__ void __launch_bounds__(kBwdThreads)
fma_chunk_bwd(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v,
              const float *__restrict__ gate, const T *__restrict__ d_out,
              const float *__restrict__ states, const float *__restrict__ dstates,
              const float *__restrict__ carry, TO *__restrict__ dq, TO *__restrict__ dk,
              TO *__restrict__ dv, float *__restrict__ dgate, Geom g)
{
    extern __shared__ __align__(16) float smem[];
    const int chunk = blockIdx.x, bh = blockIdx.y, b = bh / g.H, h = bh - b * g.H;
    const int ldk = g.dk + 4, ldv = g.dv + 4, ldp = g.C + 4;
    const int threads = blockDim.x;
    const bool over = x_over_scores(g.C, g.dk, g.dv);
    float *sLam = smem;
    float *sQ = sLam + g.C * ldk;
    float *sK = sQ + g.C * ldk;
    float *sV = sK + g.C * ldk;
    float *sG = sV + g.C * ldv;             // dO
    float *sS = sG + g.C * ldv;             // [dk][ldv]
    float *sD = sS + g.dk * ldv;            // [dk][ldv]
    float *sP = sD + g.dk * ldv;            // [C][ldp]
    float *sdP = sP + g.C * ldp;            // [C][ldp]
    float *sSeg = sS;                       // [8][dk], before the states arrive and after they are spent
    float *sX = over ? sP : sdP + g.C * ldp;              // [C][ldk]  q*dq - k*dk
    const float *sGam = sLam + (g.C - 1) * ldk;           // exp(Lam_{C-1}) once Lam has become exp(Lam)
    const size_t chunk_id = (size_t)bh * g.N + chunk;

    const Rows sRow(sV, ldv, g.dv);
    fill_rows(sRow, g, b, h, chunk);
    __syncthreads();
    // the inputs of the call: whatever produced them has completed before the kernels in front of this one started
    load_tile(sLam, ldk, gate, sRow, g.C, g.dk);
    load_tile(sV, ldv, v, sRow, g.C, g.dv);
    load_tile(sG, ldv, d_out, sRow, g.C, g.dv);
    load_tile(sQ, ldk, q, sRow, g.C, g.dk);
    load_tile(sK, ldk, k, sRow, g.C, g.dk);
    loads_done();
    __syncthreads();
    prefix_gates(sLam, ldk, g.C, g.dk, sSeg);
    make_qt_kt(sQ, sK, sLam, ldk, g.C, g.dk);
    __syncthreads();
    pdl_wait();                             // the states come from the scans in front
    pdl_launch_dependents();
    load_state(sS, ldv, states + chunk_id * g.dk * g.dv, g.dk, g.dv);
    load_state(sD, ldv, dstates + chunk_id * g.dk * g.dv, g.dk, g.dv);
    const int nb = g.C >> 2, nsc = nb * nb;
    for (int blk = threadIdx.x; blk < 2 * nsc; blk += threads) {
        const bool p = blk < nsc;           // scores, then dO V^T
        score_block(p ? sP : sdP, ldp, p ? sQ : sG, p ? ldk : ldv, p ? sK : sV, p ? ldk : ldv, g.C, p ? g.dk : g.dv, p ? blk : blk - nsc);
    }
    loads_done();
    __syncthreads();

    const int nk = grad_blocks(g.C, g.dk), nv = grad_blocks(g.C, g.dv), total = 2 * nk + nv;
    for (int base = 0; base < total; base += threads) {
        const int t = base + threadIdx.x, kind = t < nk ? 0 : t < 2 * nk ? 1 : t < total ? 2 : 3;      // uniform over a warp
        const int blk = t - kind * nk, d = kind == 2 ? g.dv : g.dk, cs = d >> 2, r0 = 8 * (blk / cs), cb = blk % cs;
        const bool on = kind < 3 && r0 < g.C;
        Acc8 a1;
        a1.zero();
        if (on) {
            if (kind == 0) {
                mm8_nn<false>(a1, sdP, ldp, r0, sK, ldk, cb, cs, r0 + 8, nullptr);        // dP Kt
                mm8_nt(a1, sG, ldv, r0, sS, ldv, cb, cs, g.dv);                           // dO S^T
            } else if (kind == 1) {
                mm8_nt(a1, sV, ldv, r0, sD, ldv, cb, cs, g.dv);                           // V D^T
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float gm = sGam[cb + j * cs];
#pragma unroll
                    for (int i = 0; i < 8; ++i) a1.v[i][j] *= gm;
                }
                mm8_tn(a1, sdP, ldp, r0, sQ, ldk, cb, cs, r0, g.C);                       // + dP^T Qt
            } else {
                mm8_tn(a1, sP, ldp, r0, sG, ldv, cb, cs, r0, g.C);                        // P^T dO
                mm8_nn<true>(a1, sK, ldk, r0, sD, ldv, cb, cs, g.dk, sGam);               // Kh D
            }
        }
        if (over) __syncthreads();          // the score tiles are spent: they become the tile of q*dq - k*dk
        if (on) {
            TO *dst = kind == 0 ? dq : kind == 1 ? dk : dv;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int row = sRow[r0 + i], o = (r0 + i) * ldk + cb;
                float r[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    r[j] = a1.v[i][j];
                    if (kind == 0) {
                        sX[o + j * cs] = sQ[o + j * cs] * r[j];
                        r[j] *= sLam[o + j * cs];
                    } else if (kind == 1) {
                        r[j] /= sLam[o + j * cs];
                    }
                }
                if (row >= 0) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) dst[(size_t)row * d + cb + j * cs] = TO(r[j]);
                }
            }
        }
        __syncthreads();                    // every block of dq comes before the same block of dk
        if (on && kind == 1) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int o = (r0 + i) * ldk + cb + j * cs;
                    sX[o] -= sK[o] * a1.v[i][j];
                }
        }
    }
    __syncthreads();
    // gate gradient: suffix sums of x down the chunk plus what later chunks carry in, the rows cut in segments
    {
        const int nseg = min(threads / g.dk, 8), rows = (g.C + nseg - 1) / nseg;
        const int seg = threadIdx.x / g.dk, c = threadIdx.x - seg * g.dk, j0 = seg * rows, j1 = min(j0 + rows, g.C);
        if (seg < nseg) {
            float run = 0.f;
#pragma unroll 8
            for (int j = j1 - 1; j >= j0; --j) {
                run += sX[j * ldk + c];
                sX[j * ldk + c] = run;
            }
            sSeg[seg * g.dk + c] = run;
        }
        __syncthreads();
        if (seg < nseg) {
            float add = carry[chunk_id * g.dk + c];
            for (int s = seg + 1; s < nseg; ++s) add += sSeg[s * g.dk + c];
            float *dst = dgate + c;
#pragma unroll 8
            for (int j = j0; j < j1; ++j) {
                const int row = sRow[j];
                const float x = sX[j * ldk + c] + add;
                if (row >= 0) dst[(size_t)row * g.dk] = x;
            }
        }
    }
}

size_t smem_state(const Geom &g, bool bwd)
{
    const size_t ldk = g.dk + 4, ldv = g.dv + 4;
    return sizeof(float) * ((size_t)g.C * ((bwd ? 3 : 2) * ldk + (bwd ? 2 : 1) * ldv) + 8 * (size_t)g.dk);
}
size_t smem_out(const Geom &g)
{
    const size_t ldk = g.dk + 4, ldv = g.dv + 4, ldp = g.C + 4;
    size_t n = (size_t)g.C * (3 * ldk + ldv) + (size_t)g.dk * ldv;
    if (g.C > g.dk) n += (size_t)g.C * ldp;
    return sizeof(float) * n;
}
size_t smem_bwd(const Geom &g)
{
    const size_t ldk = g.dk + 4, ldv = g.dv + 4, ldp = g.C + 4;
    size_t n = (size_t)g.C * (3 * ldk + 2 * ldv + 2 * ldp) + 2 * (size_t)g.dk * ldv;
    if (!x_over_scores(g.C, g.dk, g.dv)) n += (size_t)g.C * ldk;
    return sizeof(float) * n;
}
constexpr size_t kMaxSmem = 227 * 1024;
// CTAs that share a chunk where the chunks leave SMs idle: slices of the state kernel, parts of the output kernel.  Fitted to 832
// calls of 1 to 96 chunks of 16 to 128 tokens, d_k and d_v of 16 to 128: 6.1% faster on average than a CTA per chunk, the best
// choice each time 7.4%; nine calls are slower by more than 1.5% (worst 7%).  The kernel behind is launched early and wants a place
// for its CTA too, so n slices take n + 1 of them per chunk (forward: and a tenth to spare); wide heads gain as long as there are two SMs per
// chunk.  Little work is not worth the further loads.  Whole passes, d = 64, us:
//   24 chunks of 64 tokens: 20.7 with a CTA per chunk, 18.8 with four slices, 17.6 with four slices and two parts
//   74 chunks of 64: 22.2, 26.3 with two slices and two parts;  64 chunks of 32: 15.2 and 18.1;  72 chunks of 128: 43.6, 33.6 with four
//   and two;  24 chunks of 16, backward pass: 24.0, 24.0 with four slices
struct Sharing {
    int slices, parts;
};
Sharing share(const Geom &g, bool backward)
{
    const long long sms = device_sm_count(), chunks = (long long)g.N * g.B * g.H;
    auto places = [&](int per_chunk) { return per_chunk * chunks <= sms; };
    const bool wide = g.dk * g.dv > 4096, work = g.C * g.dk * g.dv > (backward ? 65536 : 32768);
    Sharing s{1, 1};
    for (int n = 4; work && n > 1 && s.slices == 1; n /= 2)
        if (g.dk % (4 * n) == 0 && (wide ? places(2) : backward ? places(n + 1) : 11 * (n + 1) * chunks <= 10 * sms)) s.slices = n;        // whole vectors of channels
    if (!backward && ((g.C == 128 || (g.C == 64 && wide)) ? places(2) : g.C == 64 && g.dv >= 48 && places(4))) {
        s.parts = 2;
        if (work && !places(3) && g.dk % 16 == 0) s.slices = 4;
    }
    return s;
}
template <typename K>
dig_status set_smem(K kernel, size_t bytes)
{
    if (bytes > kMaxSmem) return DIG_ERR_UNSUPPORTED;
    return ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), bytes);
}

template <typename T, typename TO>
dig_status fwd_typed(const GlaArgs &a)
{
    const Geom &g = a.g;
    const Workspace w = carve_workspace(a.ws, g, false);
    const Sharing shared = share(g, false);
    const dim3 grid(g.N, g.B * g.H), grid1(g.N, g.B * g.H, shared.slices);
    dig_status st;
    auto k1 = grid1.z > 1 ? fma_chunk_state<T, false, true> : fma_chunk_state<T, false, false>;
    if ((st = set_smem(k1, smem_state(g, false))) != DIG_OK) return st;
    { KernelTimer t(KID_FMA_STATE, a.stream);
    launch_pdl(k1, grid1, dim3(kThreads), smem_state(g, false), a.stream, (const T *)a.q, (const T *)a.k, (const T *)a.v, a.gate,
               (const T *)nullptr, w.states, w.gamma, (float *)nullptr, g); }
    if ((st = launch_state_scan_fwd(w, g, a.stream, a.sio)) != DIG_OK) return st;
    const int parts = shared.parts;
    auto k3 = parts > 1 ? fma_chunk_out<T, TO, 3, true>
              : g.C < 64 && (long long)grid.x * grid.y > 3ll * device_sm_count() ? fma_chunk_out<T, TO, 4, false> : fma_chunk_out<T, TO, 3, false>;
    if ((st = set_smem(k3, smem_out(g))) != DIG_OK) return st;
    KernelTimer t(KID_FMA_OUT, a.stream);
    launch_pdl(k3, dim3(grid.x, grid.y, parts), dim3(kThreads), smem_out(g), a.stream, (const T *)a.q, (const T *)a.k, (const T *)a.v, a.gate,
               (const float *)w.states, (TO *)a.out, g);
    return cuda_ok(cudaGetLastError());
}

template <typename T, typename TO>
dig_status bwd_typed(const GlaArgs &a)
{
    const Geom &g = a.g;
    const Workspace w = carve_workspace(a.ws, g, true);
    const dim3 grid(g.N, g.B * g.H), grid1(g.N, g.B * g.H, share(g, true).slices);
    dig_status st;
    auto k1 = grid1.z > 1 ? fma_chunk_state<T, true, true> : fma_chunk_state<T, true, false>;
    if ((st = set_smem(k1, smem_state(g, true))) != DIG_OK) return st;
    auto k4 = fma_chunk_bwd<T, TO>;
    if ((st = set_smem(k4, smem_bwd(g))) != DIG_OK) return st;
    { KernelTimer t(KID_FMA_STATE, a.stream);
    launch_pdl(k1, grid1, dim3(kThreads), smem_state(g, true), a.stream, (const T *)a.q, (const T *)a.k, (const T *)a.v, a.gate,
               (const T *)a.d_out, w.states, w.gamma, w.dstates, g); }
    if ((st = launch_state_scan_fwd(w, g, a.stream, a.sio)) != DIG_OK) return st;
    if ((st = launch_state_scan_bwd(w, g, a.stream, a.sio)) != DIG_OK) return st;
    KernelTimer t(KID_FMA_BWD, a.stream);
    launch_pdl(k4, grid, dim3(bwd_threads(g.C)), smem_bwd(g), a.stream, (const T *)a.q, (const T *)a.k, (const T *)a.v, a.gate,
               (const T *)a.d_out, (const float *)w.states, (const float *)w.dstates, (const float *)w.carry, (TO *)a.dq,
               (TO *)a.dk, (TO *)a.dv, a.dgate, g);
    return cuda_ok(cudaGetLastError());
}

}  // namespace

bool fma_supports(int dk, int dv, int chunk, int dtype, bool backward)
{
    (void)dtype;
    Geom g{};
    g.dk = dk; g.dv = dv; g.C = chunk;
    if (backward) return smem_bwd(g) <= kMaxSmem && smem_state(g, true) <= kMaxSmem;
    return smem_out(g) <= kMaxSmem && smem_state(g, false) <= kMaxSmem;
}

dig_status fma_gla_fwd(const GlaArgs &a)
{
    switch (a.dtype) {
        case DIG_F32: return fwd_typed<float, float>(a);
        case DIG_BF16: return fwd_typed<__nv_bfloat16, __nv_bfloat16>(a);
        case DIG_BF16_F32OUT: return fwd_typed<__nv_bfloat16, float>(a);
    }
    return DIG_ERR_INVALID_ARG;
}

dig_status fma_gla_bwd(const GlaArgs &a)
{
    switch (a.dtype) {
        case DIG_F32: return bwd_typed<float, float>(a);
        case DIG_BF16: return bwd_typed<__nv_bfloat16, __nv_bfloat16>(a);
        case DIG_BF16_F32OUT: return bwd_typed<__nv_bfloat16, float>(a);
    }
    return DIG_ERR_INVALID_ARG;
}

}  // namespace dig
