// Output gate of the GLA layer (Eq. attn_gla, the line that forms Y_t before the projection W_O):
//     z = Swish(r) (.) LN(o)      per (token, head) row of d_v values,
// and its reverse mode.  Elementwise plus two row reductions, so bandwidth-bound once the instruction count
// allows it.  Two ways, by row length and storage type (Split, below):
//   - Through shared memory.  The rows are contiguous in memory: a CTA walks over tiles of as many rows as it holds, each
//     tensor's tile fetched by one bulk copy (two tiles in flight) and the results written by one, so no thread
//     spends instructions on global addresses and every line moves once, whatever the row length.  A row is held by LPR
//     lanes with CPL neighbouring chunks of 8 values each, 4 lanes x 2 chunks up to 64 values, 3 x 3 for 72 (ten rows
//     per warp): few lanes per row keep the shuffles of the row sums small against the arithmetic.  What it is for are rows of 72:
//     the 48-byte pieces that three lanes would load share sectors, which the L1 loses when more CTAs are resident.
//   - Directly.  Every lane loads one chunk (8, 9 or 16 lanes a row).
// 262144 rows of 72 in bf16: forward 30.0 us with nine lanes of one chunk, unpacked arithmetic and loads by every
// thread, 18 us now (6.3 TB/s); reverse 54.5 -> 33.5 us (5.6 TB/s).
// The affine gradients are summed per CTA in registers and shared memory and then across CTAs by a second
// kernel in a fixed order.
// The waits for the copies are bounded like those of the sweep kernels: where one expires the rows after it stay unwritten
// and the device status word says so.
#include <type_traits>

#include "dig_common.cuh"
#include "umma.cuh"

namespace dig {
namespace {

// Threads per CTA and CTAs per SM (what the grid is capped at, so that the grid-stride loops end together): the
// forward kernel as many as shared memory holds, up to 8 (4, 5, 6 and 8 were measured: 17.7, 17.2, 16.7, 15.6 us on
// 196608 rows of 64), the reverse one 3 (2, 3, 4: 37, 33, 45 us on 262144 rows of 72), or 2 with the next row ahead.
constexpr int kThreads = 128, kFwdPerSM = 8, kBwdPerSM = 3, kAheadPerSM = 2;
constexpr size_t kSmemPerSM = 228 * 1024;

// Eight values as they are stored.
template <typename T> struct Raw8;
template <> struct Raw8<float> {
    float4 a, b;
    __device__ __forceinline__ void load(const float *p) { a = load4(p); b = load4(p + 4); }
    __device__ __forceinline__ void zero() { a = b = make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ __forceinline__ float2 pair(int j) const
    {
        return j == 0 ? make_float2(a.x, a.y) : j == 1 ? make_float2(a.z, a.w) : j == 2 ? make_float2(b.x, b.y) : make_float2(b.z, b.w);
    }
};
template <> struct Raw8<__nv_bfloat16> {
    uint4 u;
    __device__ __forceinline__ void load(const __nv_bfloat16 *p) { u = *reinterpret_cast<const uint4 *>(p); }
    __device__ __forceinline__ void zero() { u = make_uint4(0, 0, 0, 0); }
    __device__ __forceinline__ float2 pair(int j) const { return bf2(j == 0 ? u.x : j == 1 ? u.y : j == 2 ? u.z : u.w); }
};
__device__ __forceinline__ void store8(float *p, const float2 *f)
{
    store4(p, make_float4(f[0].x, f[0].y, f[1].x, f[1].y));
    store4(p + 4, make_float4(f[2].x, f[2].y, f[3].x, f[3].y));
}
__device__ __forceinline__ void store8(__nv_bfloat16 *p, const float2 *f)
{
    uint4 u;
    __nv_bfloat162 t;
    t = __float22bfloat162_rn(f[0]); u.x = *reinterpret_cast<uint32_t *>(&t);
    t = __float22bfloat162_rn(f[1]); u.y = *reinterpret_cast<uint32_t *>(&t);
    t = __float22bfloat162_rn(f[2]); u.z = *reinterpret_cast<uint32_t *>(&t);
    t = __float22bfloat162_rn(f[3]); u.w = *reinterpret_cast<uint32_t *>(&t);
    *reinterpret_cast<uint4 *>(p) = u;
}

// Arithmetic on pairs: packed instructions for bf16 rows, whose bound they are; one by one for fp32 rows, which the packed
// form slows down (196608 rows of 64 without shared memory: 19 -> 16.5 us, reverse 33 -> 32; of 8 values 14 -> 11.7 and 27 -> 22).
struct Packed {
    static __device__ __forceinline__ float2 add(float2 a, float2 b) { return add2(a, b); }
    static __device__ __forceinline__ float2 mul(float2 a, float2 b) { return mul2(a, b); }
    static __device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return fma2(a, b, c); }
};
struct Single {
    static __device__ __forceinline__ float2 add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
    static __device__ __forceinline__ float2 mul(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
    static __device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)); }
};
template <typename T> using OpsFor = std::conditional_t<sizeof(T) == 2, Packed, Single>;

// Thread -> (row slot of the CTA, lane of the row's group): 32 / LPR rows per warp.
template <int LPR, int THREADS>
struct RowMap {
    static constexpr int kRowsPerWarp = 32 / LPR, kRows = (THREADS / 32) * kRowsPerWarp;
    int lane, slot, gbase;      // lane in the group, row slot, first warp lane of the group
    bool valid;                 // false for the warp's left-over lanes when LPR is not a power of two
    __device__ __forceinline__ RowMap()
    {
        const int l = threadIdx.x & 31, grp = l / LPR;
        lane = l - grp * LPR;
        gbase = grp * LPR;
        valid = grp < kRowsPerWarp;
        slot = (threadIdx.x >> 5) * kRowsPerWarp + (valid ? grp : 0);
    }
};
// Sum over the row's lane group, returned to all of its lanes.  Power-of-two groups: butterfly.  Three
// lanes: the two others' values.  Nine lanes: the ninth is folded into the first, a butterfly over the first
// eight, then a broadcast.
template <int LPR, int THREADS> __device__ __forceinline__ float group_sum(float x, const RowMap<LPR, THREADS> &m)
{
    static_assert((LPR & (LPR - 1)) == 0 || LPR == 3 || LPR == 9, "lane groups of a power of two, of three or of nine");
    if constexpr ((LPR & (LPR - 1)) == 0) {
#pragma unroll
        for (int k = LPR / 2; k >= 1; k >>= 1) x += __shfl_xor_sync(0xffffffffu, x, k);
        return x;
    } else if constexpr (LPR == 3) {
        const float y = __shfl_sync(0xffffffffu, x, min(m.gbase + (m.lane == 2 ? 0 : m.lane + 1), 31));
        const float z = __shfl_sync(0xffffffffu, x, min(m.gbase + (m.lane == 0 ? 2 : m.lane - 1), 31));
        return x + (y + z);
    } else {
        const float y = __shfl_sync(0xffffffffu, x, min(m.gbase + 8, 31));
        if (m.lane == 0) x += y;
#pragma unroll
        for (int k = 4; k >= 1; k >>= 1) {
            const float t = __shfl_sync(0xffffffffu, x, min(m.gbase + ((m.lane ^ k) & 7), 31));
            if (m.lane < 8) x += t;
        }
        return __shfl_sync(0xffffffffu, x, m.gbase);
    }
}

// What a lane holds of a row: CPL chunks; chunk i starts at column col(i), of which ok(i) exist.
template <int LPR, int CPL, int THREADS, bool FULL>
struct Lane {
    const RowMap<LPR, THREADS> m;
    int dv;
    bool row_ok;
    // with two chunks per lane odd rows take them in the other order: the lanes of two rows then hit different banks
    __device__ __forceinline__ int col(int i) const { return 8 * (CPL * m.lane + (CPL == 2 ? i ^ (m.slot & 1) : i)); }
    __device__ __forceinline__ bool has_col(int i) const { return m.valid && (FULL || col(i) < dv); }       // FULL: LPR * CPL chunks are the row
    __device__ __forceinline__ bool ok(int i) const { return row_ok && has_col(i); }
};
template <typename T, int CPL, typename LN>
__device__ __forceinline__ void load_row(Raw8<T> (&x)[CPL], const T *p, const LN &ln)
{
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
        x[i].zero();
        if (ln.ok(i)) x[i].load(p + ln.col(i));
    }
}
// Normalised row n = (o - mean) * rstd (zero where the lane holds none).
template <typename V, typename T, int LPR, int CPL, int THREADS, bool FULL>
__device__ __forceinline__ float normalise(const Raw8<T> (&o)[CPL], const Lane<LPR, CPL, THREADS, FULL> &ln, float inv_d, float eps, float2 (&n)[4 * CPL])
{
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < CPL; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            n[4 * i + j] = o[i].pair(j);
            s = V::add(s, n[4 * i + j]);
        }
    // minus the mean as sum * (1 / d) inside a fused multiply-add: rounded on its own it costs rows far from zero (mean 16
    // deviations) three times the error
    const float sum = group_sum(s.x + s.y, ln.m);
    const float2 minus = make_float2(-sum, -sum), scale = make_float2(inv_d, inv_d);
    float2 v = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < CPL; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float2 &x = n[4 * i + j];
            x = V::fma(minus, scale, x);
            if (!FULL && !ln.has_col(i)) x = make_float2(0.f, 0.f);
            v = V::fma(x, x, v);
        }
    // slots past the last row hold zeros: with eps = 0 their 1/0 must not become 0 * inf in the affine gradients
    const float var = group_sum(v.x + v.y, ln.m) * inv_d;
    const float rstd = ln.row_ok ? rsqrtf(var + eps) : 0.f;
    const float2 sc = make_float2(rstd, rstd);
#pragma unroll
    for (int i = 0; i < 4 * CPL; ++i) n[i] = V::mul(n[i], sc);
    return rstd;
}

// 1 / (1 + e^-r) with the fast exponential and the fast reciprocal (2 ulp each; e^-r = inf gives 0)
template <typename V>
__device__ __forceinline__ float2 sigmoid2(float2 r)
{
    const float2 t = V::mul(r, make_float2(-1.4426950408889634f, -1.4426950408889634f));
    float2 e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(t.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(t.y));
    e = V::add(e, make_float2(1.f, 1.f));
    return make_float2(__fdividef(1.f, e.x), __fdividef(1.f, e.y));
}

// The affine parameters of a row in shared memory: weight (1 where absent), then bias (0).  Ends with a barrier.
template <int MAXD, int THREADS>
__device__ __forceinline__ void stage_affine(float *sh, const float *ln_w, const float *ln_b, int dv)
{
    for (int c = threadIdx.x; c < MAXD; c += THREADS) {
        sh[c] = (ln_w != nullptr && c < dv) ? ln_w[c] : 1.f;
        sh[MAXD + c] = (ln_b != nullptr && c < dv) ? ln_b[c] : 0.f;
    }
    __syncthreads();
}
__device__ __forceinline__ void pairs8(const float *p, float2 (&x)[4])
{
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
    x[0] = make_float2(a.x, a.y); x[1] = make_float2(a.z, a.w); x[2] = make_float2(b.x, b.y); x[3] = make_float2(b.z, b.w);
}

// Tiles of rows through shared memory: NIN input tensors, NOUT results, two buffers of each.  Thread 0 issues
// all copies.  Per tile: wait() for the inputs, work, then hand_over(): results of this tile leave, the
// inputs of the tile after next are asked for.  One barrier per tile.
constexpr int kStages = 2;
template <int NIN, int NOUT, int ROWS>
struct TileRing {
    char *in[NIN], *out[NOUT];          // first buffer of each tensor
    const char *src[NIN];
    char *dst[NOUT];
    int in_row[NIN], out_row[NOUT];     // bytes per row
    uint64_t *bar;
    int *status;
    long long rows;
    __device__ __forceinline__ char *in_buf(int k, int it) const { return in[k] + (it & 1) * ROWS * in_row[k]; }
    __device__ __forceinline__ char *out_buf(int k, int it) const { return out[k] + (it & 1) * ROWS * out_row[k]; }
    __device__ __forceinline__ long long first(int it) const { return ((long long)blockIdx.x + (long long)it * gridDim.x) * ROWS; }
    __device__ __forceinline__ void fetch(int it) const          // thread 0
    {
        const long long r0 = first(it);
        if (r0 >= rows) return;
        const uint32_t n = (uint32_t)(rows - r0 < ROWS ? rows - r0 : ROWS);
        uint32_t bytes = 0;
#pragma unroll
        for (int k = 0; k < NIN; ++k) bytes += n * in_row[k];
        umma::mbar_arrive_expect_tx(bar + (it & 1), bytes);
#pragma unroll
        for (int k = 0; k < NIN; ++k) umma::bulk_g2s(in_buf(k, it), src[k] + r0 * in_row[k], n * in_row[k], bar + (it & 1));
    }
    __device__ __forceinline__ bool wait(int it) const { return umma::mbar_wait(bar + (it & 1), (it >> 1) & 1, status); }
    __device__ __forceinline__ bool hand_over(int it, bool ok) const
    {
        umma::fence_async_smem();
        if (threadIdx.x == 0) umma::bulk_wait_read();            // the results of the tile before have left their buffer
        if (!__syncthreads_and(ok)) return false;
        if (threadIdx.x == 0) {
            const long long r0 = first(it);
            const uint32_t n = (uint32_t)(rows - r0 < ROWS ? rows - r0 : ROWS);
#pragma unroll
            for (int k = 0; k < NOUT; ++k) umma::bulk_s2g(dst[k] + r0 * out_row[k], out_buf(k, it), n * out_row[k]);
            umma::bulk_commit();
            fetch(it + kStages);
        }
        return true;
    }
    // After the loop: copies in flight end before the CTA's shared memory goes (also where a wait gave up at tile `it`).
    __device__ __forceinline__ void drain(int it, bool ok) const
    {
        if (threadIdx.x != 0) return;
        umma::bulk_wait_all();
        if (!ok) {
            for (int k = 0; k < kStages; ++k)
                if (first(it + k) < rows) umma::mbar_wait(bar + ((it + k) & 1), ((it + k) >> 1) & 1, status);
        }
    }
};
__device__ __forceinline__ void ring_setup(uint64_t *bar)
{
    if (threadIdx.x == 0) {
        umma::mbar_init(bar, 1);
        umma::mbar_init(bar + 1, 1);
        umma::fence_barrier_init();
    }
}

// TA: type of o (the GLA output: input storage type when it comes from memory written by a caller, output
// storage type when it comes straight from the forward pass), TR: type of r, TZ: type of z.  o and z may
// be the same buffer: a tile's rows are written after they have been read.
template <typename TA, typename TR, typename TZ, int LPR, int CPL, bool FULL>
__global__ void __launch_bounds__(kThreads)
outgate_fwd(const TA *o, const TR *r, const float *__restrict__ ln_w, const float *__restrict__ ln_b, TZ *z, long long rows,
            int dv_, float eps, int *status)
{
    constexpr int kRows = RowMap<LPR, kThreads>::kRows, kMaxD = 8 * LPR * CPL;
    extern __shared__ __align__(128) char smem[];
    __shared__ __align__(16) float aff[2 * kMaxD];
    __shared__ uint64_t bar[2];
    const int dv = FULL ? kMaxD : dv_;
    TileRing<2, 1, kRows> ring;
    ring.in_row[0] = dv * (int)sizeof(TA);
    ring.in_row[1] = dv * (int)sizeof(TR);
    ring.out_row[0] = dv * (int)sizeof(TZ);
    ring.in[0] = smem;
    ring.in[1] = ring.in[0] + kStages * kRows * ring.in_row[0];
    ring.out[0] = ring.in[1] + kStages * kRows * ring.in_row[1];
    ring.src[0] = reinterpret_cast<const char *>(o);
    ring.src[1] = reinterpret_cast<const char *>(r);
    ring.dst[0] = reinterpret_cast<char *>(z);
    ring.bar = bar;
    ring.status = status;
    ring.rows = rows;
    ring_setup(bar);
    Lane<LPR, CPL, kThreads, FULL> ln;
    ln.dv = dv;
    const float inv_d = 1.f / (float)dv;
    pdl_wait();
    if (threadIdx.x == 0) {
        ring.fetch(0);
        ring.fetch(1);
    }
    stage_affine<kMaxD, kThreads>(aff, ln_w, ln_b, dv);         // behind the wait: the kernel in front may have written them
    bool ok = true;
    int it = 0;
    for (; ok && ring.first(it) < rows; ++it) {
        ok = ring.wait(it);
        ln.row_ok = ring.first(it) + ln.m.slot < rows;
        Raw8<TA> ov[CPL];
        Raw8<TR> rv[CPL];
        load_row(ov, reinterpret_cast<const TA *>(ring.in_buf(0, it)) + ln.m.slot * dv, ln);
        load_row(rv, reinterpret_cast<const TR *>(ring.in_buf(1, it)) + ln.m.slot * dv, ln);
        float2 n[4 * CPL];
        normalise<Packed>(ov, ln, inv_d, eps, n);
        TZ *zb = reinterpret_cast<TZ *>(ring.out_buf(0, it)) + ln.m.slot * dv;
#pragma unroll
        for (int i = 0; i < CPL; ++i) {
            float2 w[4], b[4], out[4];
            pairs8(aff + ln.col(i), w);
            pairs8(aff + kMaxD + ln.col(i), b);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 x = rv[i].pair(j);
                out[j] = mul2(mul2(x, sigmoid2<Packed>(x)), fma2(n[4 * i + j], w[j], b[j]));
            }
            if (ln.ok(i)) store8(zb + ln.col(i), out);
        }
        ok = ring.hand_over(it, ok);
        if (!ok) break;
    }
    pdl_launch_dependents();
    ring.drain(it, ok);
}

// What the reverse mode keeps of a row: with n the normalised row, dy = dz Swish(r), dn = dy w,
//   dr = dz y Swish'(r),   do = rstd (dn - mean(dn) - n mean(dn n)),   dw += dy n,   db += dy.
template <typename V, int CPL>
struct RowGrad {
    float2 n[4 * CPL], dn[4 * CPL], s1, s2;
    float rstd, m1, m2;
    __device__ __forceinline__ void start(float rstd_)
    {
        rstd = rstd_;
        s1 = s2 = make_float2(0.f, 0.f);
    }
    template <typename T>
    __device__ __forceinline__ void chunk(int i, const Raw8<T> &rv, const Raw8<T> &gv, const float2 (&w)[4], const float2 (&b)[4], float2 (&aw)[4 * CPL],
                                          float2 (&ab)[4 * CPL], float2 (&dr)[4])
    {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int e = 4 * i + j;
            const float2 x = rv.pair(j), g = gv.pair(j), sg = sigmoid2<V>(x), sw = V::mul(x, sg);
            const float2 y = V::fma(n[e], w[j], b[j]), dy = V::mul(g, sw);
            dr[j] = V::mul(V::mul(g, y), V::fma(sw, V::fma(sg, make_float2(-1.f, -1.f), make_float2(1.f, 1.f)), sg));
            aw[e] = V::fma(dy, n[e], aw[e]);
            ab[e] = V::add(ab[e], dy);
            dn[e] = V::mul(dy, w[j]);
            s1 = V::add(s1, dn[e]);
            s2 = V::fma(dn[e], n[e], s2);
        }
    }
    template <typename M>
    __device__ __forceinline__ void finish(const M &m, float inv_d)
    {
        m1 = group_sum(s1.x + s1.y, m) * inv_d;
        m2 = group_sum(s2.x + s2.y, m) * inv_d;
    }
    __device__ __forceinline__ void d_o(int i, float2 (&x)[4]) const
    {
        const float2 k0 = make_float2(-rstd * m1, -rstd * m1), k1 = make_float2(-rstd * m2, -rstd * m2), k2 = make_float2(rstd, rstd);
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = V::fma(k2, dn[4 * i + j], V::fma(k1, n[4 * i + j], k0));
    }
};
// partial[cta][2][dv]: the row slots' sums of dw and db
template <int ROWS, int MAXD, int THREADS>
__device__ __forceinline__ void write_partial(const float (*red)[2][MAXD], float *partial, int dv)
{
    for (int idx = threadIdx.x; idx < 2 * MAXD; idx += THREADS) {
        const int which = idx / MAXD, c = idx - which * MAXD;
        if (c >= dv) continue;
        float sum = 0.f;
#pragma unroll 8
        for (int s = 0; s < ROWS; ++s) sum += red[s][which][c];
        partial[((size_t)blockIdx.x * 2 + which) * dv + c] = sum;
    }
}

template <typename TI, typename TO, int LPR, int CPL, bool FULL>
__global__ void __launch_bounds__(kThreads, kBwdPerSM)
outgate_bwd(const TI *o, const TI *r, const TI *dz, const float *__restrict__ ln_w, const float *__restrict__ ln_b, TO *d_o,
            TO *d_r, float *__restrict__ partial, long long rows, int dv_, float eps, int *status)
{
    constexpr int kRows = RowMap<LPR, kThreads>::kRows, kMaxD = 8 * LPR * CPL, NP = 4 * CPL;
    extern __shared__ __align__(128) char smem[];
    __shared__ __align__(16) float aff[2 * kMaxD];
    __shared__ uint64_t bar[2];
    const int dv = FULL ? kMaxD : dv_;
    TileRing<3, 2, kRows> ring;
    const char *src[3] = {reinterpret_cast<const char *>(o), reinterpret_cast<const char *>(r), reinterpret_cast<const char *>(dz)};
    char *dst[2] = {reinterpret_cast<char *>(d_o), reinterpret_cast<char *>(d_r)};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        ring.in_row[k] = dv * (int)sizeof(TI);
        ring.in[k] = smem + k * kStages * kRows * ring.in_row[k];
        ring.src[k] = src[k];
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        ring.out_row[k] = dv * (int)sizeof(TO);
        ring.out[k] = smem + 3 * kStages * kRows * ring.in_row[0] + k * kStages * kRows * ring.out_row[k];
        ring.dst[k] = dst[k];
    }
    ring.bar = bar;
    ring.status = status;
    ring.rows = rows;
    ring_setup(bar);
    Lane<LPR, CPL, kThreads, FULL> ln;
    ln.dv = dv;
    const float inv_d = 1.f / (float)dv;
    float2 aw[NP], ab[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) aw[e] = ab[e] = make_float2(0.f, 0.f);
    pdl_wait();
    if (threadIdx.x == 0) {
        ring.fetch(0);
        ring.fetch(1);
    }
    stage_affine<kMaxD, kThreads>(aff, ln_w, ln_b, dv);         // behind the wait: the kernel in front may have written them
    bool ok = true;
    int it = 0;
    for (; ok && ring.first(it) < rows; ++it) {
        ok = ring.wait(it);
        ln.row_ok = ring.first(it) + ln.m.slot < rows;
        Raw8<TI> ov[CPL], rv[CPL], gv[CPL];
        load_row(ov, reinterpret_cast<const TI *>(ring.in_buf(0, it)) + ln.m.slot * dv, ln);
        load_row(rv, reinterpret_cast<const TI *>(ring.in_buf(1, it)) + ln.m.slot * dv, ln);
        load_row(gv, reinterpret_cast<const TI *>(ring.in_buf(2, it)) + ln.m.slot * dv, ln);       // zero where the lane holds no value: it adds nothing
        TO *dob = reinterpret_cast<TO *>(ring.out_buf(0, it)) + ln.m.slot * dv, *drb = reinterpret_cast<TO *>(ring.out_buf(1, it)) + ln.m.slot * dv;
        RowGrad<Packed, CPL> g;
        g.start(normalise<Packed>(ov, ln, inv_d, eps, g.n));
#pragma unroll
        for (int i = 0; i < CPL; ++i) {
            float2 w[4], b[4], dr[4];
            pairs8(aff + ln.col(i), w);
            pairs8(aff + kMaxD + ln.col(i), b);
            g.chunk(i, rv[i], gv[i], w, b, aw, ab, dr);
            if (ln.ok(i)) store8(drb + ln.col(i), dr);
        }
        g.finish(ln.m, inv_d);
#pragma unroll
        for (int i = 0; i < CPL; ++i) {
            float2 x[4];
            g.d_o(i, x);
            if (ln.ok(i)) store8(dob + ln.col(i), x);
        }
        ok = ring.hand_over(it, ok);
        if (!ok) break;
    }
    pdl_launch_dependents();
    ring.drain(it, ok);
    if (partial == nullptr) return;
    __syncthreads();                                             // the copies have left: the ring becomes scratch
    float (*red)[2][kMaxD] = reinterpret_cast<float (*)[2][kMaxD]>(smem);
    if (ln.m.valid) {
#pragma unroll
        for (int i = 0; i < CPL; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                *reinterpret_cast<float2 *>(&red[ln.m.slot][0][ln.col(i) + 2 * j]) = aw[4 * i + j];
                *reinterpret_cast<float2 *>(&red[ln.m.slot][1][ln.col(i) + 2 * j]) = ab[4 * i + j];
            }
    }
    __syncthreads();
    write_partial<kRows, kMaxD, kThreads>(red, partial, dv);
}

// The same without shared memory: every lane loads its chunk of a row from global memory, one chunk per lane (8, 9 or 16
// lanes a row).
template <int LPR>
struct Direct {
    static constexpr int kThreads = 256, kRows = RowMap<LPR, kThreads>::kRows, kMaxD = 8 * LPR;
    using LN = Lane<LPR, 1, kThreads, false>;
};
__device__ __forceinline__ void load_affine(const float *p, int col, float absent, bool has, float2 (&x)[4])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = p != nullptr && has ? make_float2(p[col + 2 * j], p[col + 2 * j + 1]) : make_float2(absent, absent);
}
template <typename TA, typename TR, typename TZ, int LPR>
__global__ void __launch_bounds__(Direct<LPR>::kThreads, LPR == 9 ? 4 : sizeof(TR) == 2 ? 5 : 1)
outgate_fwd_direct(const TA *o, const TR *r, const float *__restrict__ ln_w, const float *__restrict__ ln_b, TZ *z, long long rows, int dv, float eps)
{
    using DR = Direct<LPR>;
    using V = OpsFor<TR>;
    typename DR::LN ln;
    ln.dv = dv;
    const int col = ln.col(0);
    const float inv_d = 1.f / (float)dv;
    pdl_wait();
    float2 w[4], b[4];
    load_affine(ln_w, col, 1.f, ln.has_col(0), w);
    load_affine(ln_b, col, 0.f, ln.has_col(0), b);
    for (long long base = (long long)blockIdx.x * DR::kRows; base < rows; base += (long long)gridDim.x * DR::kRows) {
        const long long row = base + ln.m.slot;
        ln.row_ok = row < rows;
        Raw8<TA> ov[1];
        Raw8<TR> rv[1];
        load_row(ov, o + row * dv, ln);
        load_row(rv, r + row * dv, ln);
        float2 n[4], out[4];
        normalise<V>(ov, ln, inv_d, eps, n);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 x = rv[0].pair(j);
            out[j] = V::mul(V::mul(x, sigmoid2<V>(x)), V::fma(n[j], w[j], b[j]));
        }
        if (ln.ok(0)) store8(z + row * dv + col, out);
    }
    pdl_launch_dependents();
}
template <typename TI, typename TO, int LPR, bool AHEAD>
__global__ void __launch_bounds__(Direct<LPR>::kThreads, AHEAD ? kAheadPerSM : kBwdPerSM)
outgate_bwd_direct(const TI *o, const TI *r, const TI *dz, const float *__restrict__ ln_w, const float *__restrict__ ln_b, TO *d_o, TO *d_r,
                   float *__restrict__ partial, long long rows, int dv, float eps)
{
    using DR = Direct<LPR>;
    using V = OpsFor<TI>;
    __shared__ float red[DR::kRows][2][DR::kMaxD];
    typename DR::LN ln;
    ln.dv = dv;
    const int col = ln.col(0);
    const float inv_d = 1.f / (float)dv;
    pdl_wait();
    float2 w[4], b[4], aw[4], ab[4];
    load_affine(ln_w, col, 1.f, ln.has_col(0), w);
    load_affine(ln_b, col, 0.f, ln.has_col(0), b);
#pragma unroll
    for (int j = 0; j < 4; ++j) aw[j] = ab[j] = make_float2(0.f, 0.f);
    const long long step = (long long)gridDim.x * DR::kRows;
    Raw8<TI> ov[1], rv[1], gv[1], no[1], nr[1], ng[1];
    auto load = [&](long long row, Raw8<TI> (&x)[1], Raw8<TI> (&y)[1], Raw8<TI> (&z)[1]) {
        ln.row_ok = row < rows;
        load_row(x, o + row * dv, ln);
        load_row(y, r + row * dv, ln);
        load_row(z, dz + row * dv, ln);
    };
    if (AHEAD) load((long long)blockIdx.x * DR::kRows + ln.m.slot, no, nr, ng);
    for (long long base = (long long)blockIdx.x * DR::kRows; base < rows; base += step) {
        const long long row = base + ln.m.slot;
        if (AHEAD) {
            ov[0] = no[0];
            rv[0] = nr[0];
            gv[0] = ng[0];
            load(row + step, no, nr, ng);
            ln.row_ok = row < rows;
        } else {
            load(row, ov, rv, gv);
        }
        RowGrad<V, 1> g;
        g.start(normalise<V>(ov, ln, inv_d, eps, g.n));
        float2 dr[4], dx[4];
        g.chunk(0, rv[0], gv[0], w, b, aw, ab, dr);
        if (ln.ok(0)) store8(d_r + row * dv + col, dr);
        g.finish(ln.m, inv_d);
        g.d_o(0, dx);
        if (ln.ok(0)) store8(d_o + row * dv + col, dx);
    }
    pdl_launch_dependents();
    if (partial == nullptr) return;
    if (ln.m.valid) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            *reinterpret_cast<float2 *>(&red[ln.m.slot][0][col + 2 * j]) = aw[j];
            *reinterpret_cast<float2 *>(&red[ln.m.slot][1][col + 2 * j]) = ab[j];
        }
    }
    __syncthreads();
    write_partial<DR::kRows, DR::kMaxD, DR::kThreads>(red, partial, dv);
}

// Sums of the CTAs' partial sums: lanes hold neighbouring parameters (whole lines per load), warp s of the
// block adds every kSumWarps-th partial sum, then the warps' sums are added in order (the result does not
// depend on scheduling).  One warp per parameter with lanes striding over the CTAs, each load a sector of its
// own, took about as long for 444 partial sums as this does (4.6 us, most of it launch and drain), and grew with their number.
constexpr int kSumWarps = 16;
__global__ void __launch_bounds__(32 * kSumWarps)
outgate_affine_sum(const float *__restrict__ partial, float *__restrict__ dln_w, float *__restrict__ dln_b,
                   int nctas, int dv)
{
    __shared__ float sh[kSumWarps][32];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, idx = blockIdx.x * 32 + lane;
    pdl_wait();
    pdl_launch_dependents();
    float sum = 0.f;
    if (idx < 2 * dv) {
#pragma unroll 8
        for (int s = wp; s < nctas; s += kSumWarps) sum += partial[(size_t)s * 2 * dv + idx];
    }
    sh[wp][lane] = sum;
    __syncthreads();
    if (wp != 0 || idx >= 2 * dv) return;
#pragma unroll
    for (int s = 1; s < kSumWarps; ++s) sum += sh[s][lane];
    if (idx < dv) {
        if (dln_w != nullptr) dln_w[idx] = sum;
    } else if (dln_b != nullptr) {
        dln_b[idx - dv] = sum;
    }
}

// Rows through shared memory or directly, and their split over lanes.  Measured on 196608 rows (us, through shared memory |
// directly).  Forward: bf16 rows of 72 13.6 | 19.1, of 64 12.5 | 13.5 (fp32 results 15.1 | 15.9), of 32 12.2 | 13.1 (786432 rows
// 43.8 | 52.4), of 40 13.7 | 13.4 (fp32 results 17.6 | 13.7: odd multiples of 16 bytes meet in banks), of 128 45.6 | 30.9; fp32 rows of
// 64 21.9 | 16.5, of 72 31.3 | 23.8, of 128 52.9 | 35.6.  Reverse, kernel alone, the direct one with the next row ahead: bf16 rows of
// 72 24.1 | 36.5 (fp32 results 39.6 | 42.0), of 32 19.9 | 19.4 (20.9 | 20.1), of 48 20.9 | 20.6 (25.6 | 27.7), directly of 40 19.9 (24.4), of 64
// 25.6 (32.2), of 128 50.0 (62.5); without the row ahead of 64 28.0 | 25.6 (28.3 | 31.7), of 128 92.5 | 57.2; fp32 rows of 64 46.0 | 31.9, of 72
// 63.0 | 42.9, of 128 101.8 | 58.8.  Hence shared memory for bf16 rows of 72 values and of multiples of 16 up to 64, the reverse
// mode of 64 excepted.  One rule for both result types of bf16 rows, whose results have to agree to the bit.
struct Split {
    bool ring;
    int lpr;
    Split(int dv, bool narrow, bool reverse)
        : ring(narrow && (dv == 72 || (dv <= 64 && dv % 16 == 0 && !(reverse && dv == 64)))),
          lpr(ring ? (dv == 72 ? 3 : 4) : (dv <= 64 ? 8 : dv == 72 ? 9 : 16)) {}
    int threads() const { return ring ? kThreads : Direct<8>::kThreads; }
};
// Calls f(LPR, CPL, FULL) with the split of rows that go through shared memory, or f(LPR) with that of the others.
template <bool REVERSE, typename F>
void with_ring(int dv, F f)
{
    using std::integral_constant;
    if (!REVERSE && dv == 64) f(integral_constant<int, 4>{}, integral_constant<int, 2>{}, std::bool_constant<!REVERSE>{});
    else if (dv < 64) f(integral_constant<int, 4>{}, integral_constant<int, 2>{}, std::false_type{});
    else f(integral_constant<int, 3>{}, integral_constant<int, 3>{}, std::true_type{});
}
template <typename F>
void with_direct(int dv, F f)
{
    using std::integral_constant;
    if (dv <= 64) f(integral_constant<int, 8>{});
    else if (dv == 72) f(integral_constant<int, 9>{});
    else f(integral_constant<int, 16>{});
}
int grid_for(long long rows, const Split &sp, int per_sm)
{
    int sms = device_sm_count();
    if (sms <= 0) sms = 148;            // sizing call without a device: the count the launch will most likely see
    const int kMaxCtas = sms * per_sm;
    const long long per = (sp.threads() / 32) * (32 / sp.lpr), need = (rows + per - 1) / per;
    return (int)(need < kMaxCtas ? need : kMaxCtas);
}
// Reverse mode of bf16 rows without shared memory: where a thread works more than one row, the next one is asked for before
// this one is worked.  That takes the registers of two CTAs per SM instead of three and leaves a third fewer partial sums to
// add.  Rows of 64: 196608 in a training step 28.5 -> 28.0 us and 6.1 -> 5.3 for the sums; alone, kernel and sums, 16384 rows 7.36 ->
// 6.51 (of 128: 9.30 -> 8.15), 262144 36.3 -> 35.9 (78.9 -> 68.5), but 12288 rows 6.02 -> 6.14 and 4096 3.68 -> 3.85.
bool rows_ahead(long long rows, const Split &sp, bool narrow)
{
    const long long per = (sp.threads() / 32) * (32 / sp.lpr);
    return narrow && !sp.ring && rows > grid_for(rows, sp, kBwdPerSM) * per;
}
int bwd_grid(long long rows, const Split &sp, bool narrow) { return grid_for(rows, sp, rows_ahead(rows, sp, narrow) ? kAheadPerSM : kBwdPerSM); }

template <typename TA, typename TR, typename TZ>
dig_status fwd_dispatch(const void *o, const void *r, const float *w, const float *b, void *z, long long rows, int dv,
                        float eps, cudaStream_t stream)
{
    const Split sp(dv, sizeof(TR) == 2, false);
    if constexpr (sizeof(TR) == 2) {
        if (sp.ring) {
            int *status = device_status_ptr();
            if (!status) return DIG_ERR_CUDA;
            dig_status st = DIG_OK;
            with_ring<false>(dv, [&](auto lpr, auto cpl, auto full) {
                constexpr int LPR = decltype(lpr)::value, CPL = decltype(cpl)::value, ROWS = RowMap<LPR, kThreads>::kRows;
                auto kern = outgate_fwd<TA, TR, TZ, LPR, CPL, decltype(full)::value>;
                const size_t smem = (size_t)kStages * ROWS * dv * (sizeof(TA) + sizeof(TR) + sizeof(TZ));
                if ((st = ensure_dynamic_smem(reinterpret_cast<const void *>(kern), smem)) != DIG_OK) return;
                const int fit = (int)(kSmemPerSM / (smem + 3072));           // + 1 KB of the system's and the static arrays
                const int per_sm = fit < 1 ? 1 : fit < kFwdPerSM ? fit : kFwdPerSM;
                launch_pdl(kern, dim3(grid_for(rows, sp, per_sm)), dim3(kThreads), smem, stream, (const TA *)o, (const TR *)r, w, b,
                           (TZ *)z, rows, dv, eps, status);
                st = cuda_ok(cudaGetLastError());
            });
            return st;
        }
    }
    with_direct(dv, [&](auto lpr) {
        launch_pdl(outgate_fwd_direct<TA, TR, TZ, decltype(lpr)::value>, dim3(grid_for(rows, sp, kFwdPerSM)), dim3(sp.threads()), 0, stream,
                   (const TA *)o, (const TR *)r, w, b, (TZ *)z, rows, dv, eps);
    });
    return cuda_ok(cudaGetLastError());
}

template <typename TI, typename TO>
dig_status bwd_dispatch(const void *o, const void *r, const void *dz, const float *w, const float *b, void *d_o, void *d_r,
                        float *partial, long long rows, int dv, float eps, cudaStream_t stream)
{
    const Split sp(dv, sizeof(TI) == 2, true);
    if constexpr (sizeof(TI) == 2) {
        if (sp.ring) {
            int *status = device_status_ptr();
            if (!status) return DIG_ERR_CUDA;
            dig_status st = DIG_OK;
            with_ring<true>(dv, [&](auto lpr, auto cpl, auto full) {
                constexpr int LPR = decltype(lpr)::value, CPL = decltype(cpl)::value, ROWS = RowMap<LPR, kThreads>::kRows;
                auto kern = outgate_bwd<TI, TO, LPR, CPL, decltype(full)::value>;
                const size_t ring = (size_t)kStages * ROWS * dv * (3 * sizeof(TI) + 2 * sizeof(TO)), red = (size_t)ROWS * 2 * 8 * LPR * CPL * sizeof(float);
                const size_t smem = ring > red ? ring : red;
                if ((st = ensure_dynamic_smem(reinterpret_cast<const void *>(kern), smem)) != DIG_OK) return;
                launch_pdl(kern, dim3(grid_for(rows, sp, kBwdPerSM)), dim3(kThreads), smem, stream, (const TI *)o, (const TI *)r,
                           (const TI *)dz, w, b, (TO *)d_o, (TO *)d_r, partial, rows, dv, eps, status);
                st = cuda_ok(cudaGetLastError());
            });
            return st;
        }
    }
    with_direct(dv, [&](auto lpr) {
        auto kern = outgate_bwd_direct<TI, TO, decltype(lpr)::value, false>;
        if constexpr (sizeof(TI) == 2) {
            if (rows_ahead(rows, sp, true)) kern = outgate_bwd_direct<TI, TO, decltype(lpr)::value, true>;
        }
        launch_pdl(kern, dim3(bwd_grid(rows, sp, sizeof(TI) == 2)), dim3(sp.threads()), 0, stream, (const TI *)o, (const TI *)r, (const TI *)dz, w, b,
                   (TO *)d_o, (TO *)d_r, partial, rows, dv, eps);
    });
    return cuda_ok(cudaGetLastError());
}

}  // namespace

// the wider of the two storage types' grids
size_t outgate_bwd_workspace_bytes(long long rows, int dv)
{
    const int a = grid_for(rows, Split(dv, true, true), kBwdPerSM), b = grid_for(rows, Split(dv, false, true), kBwdPerSM);
    return (size_t)(a > b ? a : b) * 2 * (size_t)dv * sizeof(float);
}

dig_status launch_outgate_fwd(const void *o, const void *r, const float *ln_w, const float *ln_b, void *z,
                              long long rows, int dv, float eps, int dtype, cudaStream_t stream)
{
    using bf16 = __nv_bfloat16;
    KernelTimer t(KID_OUTGATE, stream);
    if (dtype == DIG_F32) return fwd_dispatch<float, float, float>(o, r, ln_w, ln_b, z, rows, dv, eps, stream);
    if (dtype == DIG_BF16) return fwd_dispatch<bf16, bf16, bf16>(o, r, ln_w, ln_b, z, rows, dv, eps, stream);
    return fwd_dispatch<bf16, bf16, float>(o, r, ln_w, ln_b, z, rows, dv, eps, stream);
}

// o in the output storage type of `dtype` (as the forward pass writes it), r in the input storage type.
dig_status launch_outgate_fwd_mixed(const void *o, const void *r, const float *ln_w, const float *ln_b, void *z,
                                    long long rows, int dv, float eps, int dtype, cudaStream_t stream)
{
    if (dtype != DIG_BF16_F32OUT) return launch_outgate_fwd(o, r, ln_w, ln_b, z, rows, dv, eps, dtype, stream);
    KernelTimer t(KID_OUTGATE, stream);
    return fwd_dispatch<float, __nv_bfloat16, float>(o, r, ln_w, ln_b, z, rows, dv, eps, stream);
}

dig_status launch_outgate_bwd(const void *o, const void *r, const void *dz, const float *ln_w, const float *ln_b,
                              void *d_o, void *d_r, float *dln_w, float *dln_b, long long rows, int dv, float eps,
                              int dtype, float *partial, cudaStream_t stream)
{
    using bf16 = __nv_bfloat16;
    const bool affine = dln_w != nullptr || dln_b != nullptr;
    float *part = affine ? partial : nullptr;
    dig_status st;
    {
        KernelTimer t(KID_OUTGATE, stream);
        if (dtype == DIG_F32) st = bwd_dispatch<float, float>(o, r, dz, ln_w, ln_b, d_o, d_r, part, rows, dv, eps, stream);
        else if (dtype == DIG_BF16) st = bwd_dispatch<bf16, bf16>(o, r, dz, ln_w, ln_b, d_o, d_r, part, rows, dv, eps, stream);
        else st = bwd_dispatch<bf16, float>(o, r, dz, ln_w, ln_b, d_o, d_r, part, rows, dv, eps, stream);
    }
    if (st != DIG_OK || !affine) return st;
    KernelTimer t(KID_OUTGATE, stream);
    launch_pdl(outgate_affine_sum, dim3((2 * dv + 31) / 32), dim3(32 * kSumWarps), 0, stream, (const float *)partial, dln_w,
               dln_b, bwd_grid(rows, Split(dv, dtype != DIG_F32, true), dtype != DIG_F32), dv);
    return cuda_ok(cudaGetLastError());
}

}  // namespace dig
