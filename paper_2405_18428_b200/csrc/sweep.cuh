// Building blocks of the tcgen05 "sweep" kernels for chunkwise gated linear attention (Eq. attn_gla
// evaluated chunk by chunk, Section 3.5).  A CTA walks over consecutive 64-token tiles of one
// (batch, head) sequence and keeps the d_k x d_v state of the recurrence in registers, so per-chunk
// states never travel through memory in the forward pass.
//
// Operand tiles are fp16 (11 significant bits, like tf32, at half the bytes and with one copy
// serving both operand orientations).  fp16's narrow exponent is handled by centring the in-chunk
// decay: with Lam the cumulative gate inside a (sub-)chunk and c = Lam_end / 2 per channel, the
// tiles hold q*exp(Lam - c) and k*exp(c - Lam), whose factors stay within exp(+-|Lam_end|/2).  A
// tile whose gates sum to more than kSubLimit is worked in shorter sub-chunks of 32, 16 or 8 rows,
// each with its own centring: two of 32 in one pass over the tile where the kernel has the code for it,
// otherwise a pass each with the other rows zero.  Conversions saturate instead of overflowing.
//
// Tile layout: no swizzle, "chunk-major": element (row, col) of a tile with R rows sits at
//   (col / 8) * (16 R + 16) + 16 row + 2 (col % 8)
// i.e. 8-column chunks of 16 bytes per row, rows contiguous within a chunk, one 16-byte pad per
// chunk.  Every 8 x 16-byte core matrix is contiguous, which is what the non-swizzled tcgen05
// matrix descriptors want in both orientations, any number of columns that is a multiple of 8
// works, and both a warp that stores 32 rows of one chunk and a warp that stores the chunks of 4
// rows touch 32 different banks.
#pragma once

#include <cuda_fp16.h>

#include "dig_common.cuh"
#include "umma.cuh"

namespace dig {
namespace sw {

using namespace umma;
using bf16 = __nv_bfloat16;

constexpr int T = 64;                       // rows (scan positions) of a tile
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kSubLimit = 23.0f;          // largest |sum of gates| (log2 units, = 15.9 nats) of one (sub-)chunk
constexpr int kMinSub = 8;                  // shortest sub-chunk
constexpr int kSlots = T / kMinSub;         // sub-chunks a tile can have
constexpr int kStatusTimeout = 1, kStatusRange = 2;

template <int D>
struct Cfg {
    static_assert(D % 8 == 0 && D >= 16 && D <= 128, "head size");
    static constexpr int NCH = D / 8;               // 8-column chunks that hold data
    static constexpr int KS = (D + 15) / 16;        // MMA steps of a contraction over the channels
    static constexpr int NCHP = 2 * KS;             // chunks a tile provides (a last zero chunk pads odd counts)
    static constexpr int RS = 16 * KS;              // rows of a state tile (zero rows beyond D)
    static constexpr int CHT = T * 16 + 16;         // chunk stride of a token tile (64 rows)
    static constexpr int CHS = RS * 16 + 16;        // chunk stride of a state tile (RS rows)
    static constexpr int TILE_T = NCHP * CHT, TILE_S = NCHP * CHS, TILE_P = (T / 8) * CHT;
};

struct Plan {
    int ntile;      // 64-token tiles per sequence
    int nseg;       // segments per sequence (one CTA sweeps one segment)
    int G;          // tiles per segment
    int sub_max;    // longest sub-chunk allowed (the requested chunk size, at most 64)
    uint32_t gh_inv;// floor(2^32 / grid_h): column orders divide scan positions by the grid height
};

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Two floats -> packed fp16 (first argument in the low half), round to nearest, saturating to the
// largest finite value instead of overflowing to infinity.
__device__ __forceinline__ uint32_t pack_h2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint4 pack_h8(const float (&f)[8])
{
    return make_uint4(pack_h2(f[0], f[1]), pack_h2(f[2], f[3]), pack_h2(f[4], f[5]), pack_h2(f[6], f[7]));
}
__device__ __forceinline__ void ld8(const float *p, float (&f)[8])
{
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}
__device__ __forceinline__ void st8(float *p, const float (&f)[8])
{
    *reinterpret_cast<float4 *>(p) = make_float4(f[0], f[1], f[2], f[3]);
    *reinterpret_cast<float4 *>(p + 4) = make_float4(f[4], f[5], f[6], f[7]);
}
// 8 results to global memory in the output storage type.  `add`: on top of what is there (fp32 outputs only;
// used when several scan orders are summed into one buffer).  The addition is left to the L2 (a vector
// reduction): every element of a buffer gets one addition per launch and the launches follow one another on
// the stream, so the sum does not depend on scheduling, and nothing waits for the old values.
__device__ __forceinline__ void store_out8(float *p, const float (&f)[8], bool add = false)
{
    if (add) {
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" :: "l"(p), "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]) : "memory");
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" :: "l"(p + 4), "f"(f[4]), "f"(f[5]), "f"(f[6]), "f"(f[7]) : "memory");
    } else {
        st8(p, f);
    }
}
__device__ __forceinline__ void store_out8(bf16 *p, const float (&f)[8], bool = false)
{
    uint4 u;
    __nv_bfloat162 t;
    t = __floats2bfloat162_rn(f[0], f[1]); u.x = *reinterpret_cast<uint32_t *>(&t);
    t = __floats2bfloat162_rn(f[2], f[3]); u.y = *reinterpret_cast<uint32_t *>(&t);
    t = __floats2bfloat162_rn(f[4], f[5]); u.z = *reinterpret_cast<uint32_t *>(&t);
    t = __floats2bfloat162_rn(f[6], f[7]); u.w = *reinterpret_cast<uint32_t *>(&t);
    *reinterpret_cast<uint4 *>(p) = u;
}

// ---- matrix descriptors of chunk-major tiles -----------------------------------------------------
// K-major view (tile rows = M or N index, contraction along the columns): the two 8-column chunks
// of a 16-wide step are `ch` bytes apart (leading offset), 8-row groups 128 bytes (stride offset).
// MN-major view (tile rows = contraction index, columns = M or N index): 8-row groups along the
// contraction 128 bytes apart (leading offset), 8-column chunks along M / N `ch` bytes (stride).
__device__ __forceinline__ uint64_t kdesc(uint32_t saddr, uint32_t ch) { return make_desc(saddr, ch, 128, 0); }
__device__ __forceinline__ uint64_t mdesc(uint32_t saddr, uint32_t ch) { return make_desc(saddr, 128, ch, 0); }

// D[tmem] (+)= A * B over KSTEPS steps of 16 along the contraction.  a / b: shared-memory address
// of the first element the product uses (a row or chunk offset selects a slice), ach / bch: chunk
// strides of the tiles (compile-time, so every descriptor is the first one plus a constant in its
// low word: shared-memory addresses stay below 2^18, the address field cannot carry into the next).
// BSBO: distance of the 8-row groups of a K-major B (256 takes every other group).  SKIP: quarters of the
// accumulator's lanes that stay as they are (rows 16 q .. 16 q + 15 of an M = 64 product are in quarter q).
template <int M, int N, bool A_MN, bool B_MN, int KSTEPS, uint32_t ACH, uint32_t BCH, uint32_t BSBO, class F>
__device__ __forceinline__ void each_step(uint32_t a, uint32_t b, F mma)
{
    static_assert(M == 64 && N % 8 == 0, "instruction shape");
    constexpr uint32_t idesc = idesc_f16(M, N, A_MN, B_MN);
    const uint64_t da = A_MN ? mdesc(a, ACH) : kdesc(a, ACH), db = B_MN ? mdesc(b, BCH) : make_desc(b, BCH, BSBO, 0);
    constexpr uint32_t sa = A_MN ? 16u : (2u * ACH) >> 4, sb = B_MN ? 16u : (2u * BCH) >> 4;
    const uint32_t alo = (uint32_t)da, ahi = (uint32_t)(da >> 32), blo = (uint32_t)db, bhi = (uint32_t)(db >> 32);
#pragma unroll
    for (int kk = 0; kk < KSTEPS; ++kk) mma(kk, ((uint64_t)ahi << 32) | (alo + kk * sa), ((uint64_t)bhi << 32) | (blo + kk * sb), idesc);
}
template <int M, int N, bool A_MN, bool B_MN, int KSTEPS, uint32_t ACH, uint32_t BCH, uint32_t BSBO = 128, uint32_t SKIP = 0>
__device__ __forceinline__ void issue(uint32_t d_tmem, uint32_t a, uint32_t b, bool accumulate)
{
    each_step<M, N, A_MN, B_MN, KSTEPS, ACH, BCH, BSBO>(a, b, [&](int kk, uint64_t xa, uint64_t xb, uint32_t idesc) {
        if constexpr (SKIP == 0) mma_f16(d_tmem, xa, xb, idesc, accumulate || kk > 0);
        else mma_f16_part<SKIP>(d_tmem, xa, xb, idesc, accumulate || kk > 0);
    });
}
// D += A * B with the 64 x 64 lower triangle A (TRANSPOSED: upper), in as many instructions: where half of A's rows are zero along
// half of the contraction, they keep what they hold.  Zeros would do but for NaN, which they spread: where the halves are
// sub-chunks, to rows that do not depend on it (in the other direction the state carries a NaN over in any case).
template <int N, bool TRANSPOSED, uint32_t ACH, uint32_t BCH>
__device__ __forceinline__ void issue_triangle(uint32_t d_tmem, uint32_t a, uint32_t b)
{
    each_step<64, N, TRANSPOSED, true, T / 16, ACH, BCH, 128>(a, b, [&](int kk, uint64_t xa, uint64_t xb, uint32_t idesc) {
        if (TRANSPOSED != (kk < T / 32)) mma_f16(d_tmem, xa, xb, idesc, true);
        else mma_f16_part<TRANSPOSED ? 0xcu : 0x3u>(d_tmem, xa, xb, idesc, true);
    });
}

struct Ctl {
    uint64_t bar[4];
    uint32_t tmem_base;
    uint32_t pad;
};

// Element offset of the (batch b, head h) row of the token at scan position 64*tile + row in a
// [B][L][H][D] tensor; positions past the end of the sequence give its first row (what is read there is
// cleared).  The host checks that offsets fit 31 bits.
__device__ __forceinline__ int tile_row_offset(const Geom &g, const Plan &pl, int dir, int b, int h, int d, int tile, int row)
{
    int p = tile * T + row;
    if (p >= g.L) p = 0;
    if (dir & 1) p = g.L - 1 - p;
    if (dir & 2) {
        // p / gh with a reciprocal rounded down: the estimate is at most one too small for p < 2^24
        int x = (int)__umulhi((uint32_t)p, pl.gh_inv), y = p - x * g.gh;
        if (y >= g.gh) { y -= g.gh; ++x; }
        p = y * g.gw + x;
    }
    return ((b * g.L + p) * g.H + h) * d;
}

// Zero-fills shared memory with the CTA's threads.
__device__ __forceinline__ void zero_smem(char *p, int bytes)
{
    for (int i = threadIdx.x * 16; i < bytes; i += blockDim.x * 16) *reinterpret_cast<uint4 *>(p + i) = make_uint4(0, 0, 0, 0);
}

}  // namespace sw

// Host side of the sweep family (gla_sweep.cu).
bool sweep_supports(int dk, int dv, int chunk, int dtype);
size_t sweep_workspace_bytes(const Geom &g, bool backward);
dig_status sweep_gla_fwd(const GlaArgs &a);
dig_status sweep_gla_bwd(const GlaArgs &a);
// Sums over the scan orders of `mask` (bit d = direction d); outputs in the storage type of a.dtype.
size_t sweep_multi_workspace_bytes(const Geom &g, bool backward, int dtype);
dig_status sweep_gla_fwd_multi(const GlaArgs &a, unsigned mask);
dig_status sweep_gla_bwd_multi(const GlaArgs &a, unsigned mask);

}  // namespace dig
