// SREM depthwise 3x3 convolution (Algorithm 1: DWConv2d on the reshaped token matrix), channel-last.
// A CTA stages a (TY+2) x (TX+2) pixel halo tile of CH channels in shared memory with 16-byte
// coalesced loads; each thread then owns 8 channels of one tile column and walks down the rows.
// The scan order the residual stream is in (`dir`) only permutes the filter taps:
// reverse orders see the filter rotated by 180 degrees, column orders see it transposed.
#include <type_traits>

#include "dig_common.cuh"

namespace dig {
namespace {

constexpr int TY = 4, TX = 8, VEC = 8;
// Channels per CTA: 256 bytes of one pixel, so the halo tile stays under 48 KB of shared memory.
template <typename T> struct Cfg {
    static constexpr int CH = 256 / (int)sizeof(T);
    static constexpr int kLanes = CH / VEC;          // 16-byte (bf16) / 32-byte (fp32) vectors per pixel
    static constexpr int kThreads = kLanes * TX;
};

template <typename T> struct Vec8;
template <> struct Vec8<float> {
    float4 a, b;
    __device__ static Vec8 load(const float *p) { return {load4(p), load4(p + 4)}; }
    __device__ static Vec8 zero() { return {make_float4(0, 0, 0, 0), make_float4(0, 0, 0, 0)}; }
    __device__ void unpack(float (&f)[8]) const { f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w; }
};
template <> struct Vec8<__nv_bfloat16> {
    uint4 u;
    __device__ static Vec8 load(const __nv_bfloat16 *p) { return {*reinterpret_cast<const uint4 *>(p)}; }
    __device__ static Vec8 zero() { return {make_uint4(0, 0, 0, 0)}; }
    __device__ void unpack(float (&f)[8]) const
    {
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[2 * i] = __uint_as_float(w[i] << 16);
            f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
};

__device__ __forceinline__ void store8(float *p, const float (&f)[8])
{
    store4(p, make_float4(f[0], f[1], f[2], f[3]));
    store4(p + 4, make_float4(f[4], f[5], f[6], f[7]));
}
__device__ __forceinline__ void store8(__nv_bfloat16 *p, const float (&f)[8])
{
    uint4 u;
    __nv_bfloat162 t;
    t = __floats2bfloat162_rn(f[0], f[1]); u.x = *reinterpret_cast<uint32_t *>(&t);
    t = __floats2bfloat162_rn(f[2], f[3]); u.y = *reinterpret_cast<uint32_t *>(&t);
    t = __floats2bfloat162_rn(f[4], f[5]); u.z = *reinterpret_cast<uint32_t *>(&t);
    t = __floats2bfloat162_rn(f[6], f[7]); u.w = *reinterpret_cast<uint32_t *>(&t);
    *reinterpret_cast<uint4 *>(p) = u;
}

template <typename T, typename TO>
__global__ void __launch_bounds__(Cfg<T>::kThreads)
srem_dwconv3x3(const T *__restrict__ x, const T *__restrict__ w, const T *__restrict__ bias,
               TO *__restrict__ y, int gh, int gw, int D, int nchb, int dir)
{
    constexpr int CH = Cfg<T>::CH, kLanes = Cfg<T>::kLanes, kConvThreads = Cfg<T>::kThreads;
    __shared__ Vec8<T> tile[TY + 2][TX + 2][kLanes];
    const int b = blockIdx.z / nchb, chb = blockIdx.z - b * nchb;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int lane = threadIdx.x % kLanes, col = threadIdx.x / kLanes;
    const int ch = chb * CH + lane * VEC;
    const bool ch_ok = ch < D;
    const T *xb = x + (size_t)b * gh * gw * D;
    pdl_wait();
    pdl_launch_dependents();      // only once this kernel's own predecessor has completed

    for (int idx = threadIdx.x; idx < (TY + 2) * (TX + 2) * kLanes; idx += kConvThreads) {
        const int l = idx % kLanes, pix = idx / kLanes;
        const int tx = pix % (TX + 2), ty = pix / (TX + 2);
        const int gy = y0 + ty - 1, gx = x0 + tx - 1, c = chb * CH + l * VEC;
        Vec8<T> v = Vec8<T>::zero();
        if (gy >= 0 && gy < gh && gx >= 0 && gx < gw && c < D)
            v = Vec8<T>::load(xb + ((size_t)gy * gw + gx) * D + c);
        tile[ty][tx][l] = v;
    }
    // filter taps for this thread's channels, re-oriented: wt[u][v] multiplies x[i+u-1][j+v-1].  They are
    // kept packed (and unpacked at every use) so that the kernel stays at a register count that lets
    // six CTAs share an SM; the loads of the tile are what it waits for, not the arithmetic.
    Vec8<T> wt[3][3];
    float bs[8];
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            int su = u, sv = v;
            if (dir & 2) { su = v; sv = u; }
            if (dir & 1) { su = 2 - su; sv = 2 - sv; }
            wt[u][v] = ch_ok ? Vec8<T>::load(w + (size_t)(su * 3 + sv) * D + ch) : Vec8<T>::zero();
        }
#pragma unroll
    for (int i = 0; i < 8; ++i) bs[i] = 0.f;
    if (bias != nullptr && ch_ok) Vec8<T>::load(bias + ch).unpack(bs);
    __syncthreads();
    if (!ch_ok || x0 + col >= gw) return;

#pragma unroll
    for (int ty = 0; ty < TY; ++ty) {
        if (y0 + ty < gh) {
            float acc[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = bs[i];
#pragma unroll
            for (int u = 0; u < 3; ++u)
#pragma unroll
                for (int v = 0; v < 3; ++v) {
                    float xv[8], wv[8];
                    tile[ty + u][col + v][lane].unpack(xv);
                    wt[u][v].unpack(wv);
#pragma unroll
                    for (int i = 0; i < 8; ++i) acc[i] = fmaf(wv[i], xv[i], acc[i]);
                }
            store8(y + (((size_t)b * gh + y0 + ty) * gw + x0 + col) * D + ch, acc);
        }
    }
}

// The same convolution for grids that fill the machine, and its reverse mode.  A CTA walks down a strip of TX
// pixel columns and CH channels, row by row.  Input rows (TX + 2 pixels with the halo) arrive through cp.async in
// a ring of kRing rows, kRing - 1 rows ahead of the arithmetic, so every input row is fetched once per strip.  A
// thread owns 2 channels of four neighbouring columns: it widens the six pixels around them once per row and feeds
// the three output rows around that row from registers (o[r % 3] belongs to output row r).  Out-of-grid pixels and
// channels are zero-filled by the copy itself (source size 0).  One barrier per row: the slot refilled after the
// barrier of row r is the one row r - 1 was read from.  CTA y of a channel block takes the strips y, y + gridDim.y,
// ...; strip = (batch * strips_x + strip column) * nseg + row segment of seg_rows output rows.
//
// Reverse mode (BWD): the rows are those of dy.  With G the value of dy under tap (u, v) of the window around a pixel,
//   dx[i][j]    = sum over taps of w[2-u][2-v] G,        dw[2-u][2-v] = sum over pixels of x[i][j] G,
// so one pass over x and dy gives both; dbias = sum of dy.  Rows of x arrive beside those of dy, and dy row r meets
// the x rows r + 1, r, r - 1 (in registers, xr[r % 3]).  At the end the CTA's column groups are summed through shared
// memory and one partial sum per CTA is written; a second kernel adds the partial sums in a fixed order, so the result
// does not depend on scheduling.  A CTA reads x of its own row segment only (segments share halo rows of dy).
//
// Bound by the instructions of few warps (a fifth of the warps keep the issue slots half busy, waiting for the math pipe and for
// fixed latencies; the multiply-adds are two fifths of the instructions), then by memory: hence packed
// multiply-adds on channel pairs and one pointer per copied vector that only moves from row to row; deeper rings and
// more CTAs per SM change nothing.  128 x 128 pixels of 1152 channels in bf16: 22.5 -> 21 us forward; reverse mode in
// one pass 34 us, where dx and the filter sums in a pass each took 21 + 25.5.
constexpr int kRing = 6;
constexpr int kStripCtas = 4;        // per SM: what 128 registers allow (five at 100 registers were no faster)
constexpr int kWgPixels = 32;        // pixels per partial sum at least

__device__ __forceinline__ float2 load_pair(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ float2 load_pair(const __nv_bfloat16 *p) { return bf2(*reinterpret_cast<const uint32_t *>(p)); }
__device__ __forceinline__ void store_pair(float *p, float2 v) { *reinterpret_cast<float2 *>(p) = v; }
__device__ __forceinline__ void store_pair(__nv_bfloat16 *p, float2 v) { *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(v.x, v.y); }

// Stored tap that scan order `dir` puts at (u, v).
__device__ __forceinline__ int stored_tap(int u, int v, int dir)
{
    int su = dir & 2 ? v : u, sv = dir & 2 ? u : v;
    if (dir & 1) { su = 2 - su; sv = 2 - sv; }
    return su * 3 + sv;
}

template <typename T, typename TO, bool BWD>
__global__ void __launch_bounds__(Cfg<T>::kThreads, kStripCtas)
srem_dwconv3x3_strip(const T *__restrict__ src, const T *__restrict__ w, const T *__restrict__ bias, TO *__restrict__ dst,
                     const T *__restrict__ x, float *__restrict__ partial, int B, int gh, int gw, int D, int dir, int strips_x,
                     int nseg, int seg_rows, int nstrips)
{
    constexpr int CH = Cfg<T>::CH, kLanes = Cfg<T>::kLanes, kConvThreads = Cfg<T>::kThreads;
    constexpr int kPieces = (int)sizeof(Vec8<T>) / 16, kPairs = CH / 2, kCols = 4, kGroups = TX / kCols;
    static_assert(kPairs * kGroups == kConvThreads, "one thread per (column group, channel pair)");
    constexpr int kRowS = (TX + 2) * kLanes, kRowX = BWD ? TX * kLanes : 0, kRowVecs = kRowS + kRowX;   // vectors of a row (pair)
    constexpr int kFill = (kRowVecs + kConvThreads - 1) / kConvThreads;
    // rings of source rows and x rows; the same memory later holds the column groups' sums [groups][10][CH]
    constexpr size_t kRingBytes = sizeof(Vec8<T>) * kRing * kRowVecs;
    static_assert(!BWD || sizeof(float) * kGroups * 10 * CH <= kRingBytes, "the sums lie over the rings");
    __shared__ __align__(16) char sm[kRingBytes];
    constexpr uint32_t kSlot = sizeof(Vec8<T>) * kRowVecs, kXOff = sizeof(Vec8<T>) * kRowS;     // a slot: source row, then x row
    const int pair = threadIdx.x % kPairs, grp = threadIdx.x / kPairs, c0 = kCols * grp;
    const int chb = blockIdx.x, ch = chb * CH + 2 * pair;
    const bool ch_ok = ch < D;
    const size_t row_elems = (size_t)gw * D;
    if (BWD) dir ^= 1;                  // the taps of dx
    pdl_wait();
    float2 wf[3][3], bs = make_float2(0.f, 0.f), acc[3][3], accb = make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            wf[u][v] = ch_ok ? load_pair(w + (size_t)stored_tap(u, v, dir) * D + ch) : make_float2(0.f, 0.f);
            acc[u][v] = make_float2(0.f, 0.f);
        }
    if (!BWD && bias != nullptr && ch_ok) bs = load_pair(bias + ch);
    for (int s = blockIdx.y; s < nstrips; s += gridDim.y) {
        const int sg = s % nseg, s1 = s / nseg, sx = s1 % strips_x, b = s1 / strips_x;
        const int x0 = sx * TX, ys = sg * seg_rows, ye = min(ys + seg_rows, gh), nr = ye - ys + 2;
        const int ncol = ch_ok ? min(gw - x0 - c0, kCols) : 0;      // this thread's columns inside the grid
        // this thread's vectors of a row: source of the next copy (a valid address also where nothing is copied),
        // place in slot 0, bytes
        const T *f_src[kFill];
        uint32_t f_dst[kFill];
        int f_bytes[kFill];
        bool f_isx[kFill];
#pragma unroll
        for (int i = 0; i < kFill; ++i) {
            const int idx = (int)threadIdx.x + i * kConvThreads;
            const bool isx = BWD && (i + 1) * kConvThreads > kRowS && idx >= kRowS;
            const int j = isx ? idx - kRowS : idx, l = j % kLanes, tx = j / kLanes;
            const int gx = isx ? x0 + tx : x0 + tx - 1, c = chb * CH + l * VEC;
            const bool ok = idx < kRowVecs && gx >= 0 && gx < gw && c < D;
            f_isx[i] = isx;
            f_bytes[i] = ok ? 16 : 0;
            f_dst[i] = (uint32_t)__cvta_generic_to_shared(sm) + (uint32_t)sizeof(Vec8<T>) * idx;
            f_src[i] = (isx ? x : src) + ((size_t)b * gh + (isx ? ys : max(ys - 1, 0))) * row_elems + (ok ? (size_t)gx * D + c : 0);
        }
        auto fill = [&](int rr, uint32_t slot) {    // source row rr of the strip (image row ys - 1 + rr), x row rr (image row ys + rr)
            const int gy = ys - 1 + rr;
            const bool oks = gy >= 0 && gy < gh, okx = gy + 1 < ye;
            const size_t adv_s = gy >= 0 && gy + 1 < gh ? row_elems : 0, adv_x = gy + 2 < ye ? row_elems : 0;
#pragma unroll
            for (int i = 0; i < kFill; ++i) {
                if (i + 1 < kFill || (int)threadIdx.x + i * kConvThreads < kRowVecs) {
                    const int bytes = (f_isx[i] ? okx : oks) ? f_bytes[i] : 0;
#pragma unroll
                    for (int p = 0; p < kPieces; ++p)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(f_dst[i] + slot + 16 * p),
                                     "l"(reinterpret_cast<const char *>(f_src[i]) + 16 * p), "r"(bytes) : "memory");
                }
                f_src[i] += f_isx[i] ? adv_x : adv_s;
            }
        };
        __syncthreads();                // the previous strip's last rows have been read
#pragma unroll
        for (int i = 0; i < kRing - 1; ++i) {
            if (i < nr) fill(i, i * kSlot);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        uint32_t rd = 0, wr = (kRing - 1) * kSlot;      // slots of the row read next and of the row fetched next
        float2 o[3][kCols], xr[3][kCols];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int p = 0; p < kCols; ++p) o[r][p] = xr[r][p] = make_float2(0.f, 0.f);
        TO *orow = dst + (((size_t)b * gh + ys) * gw + x0 + c0) * D + ch;      // output row completed next
        // One input row: PH = rr % 3 is a compile-time constant so that the rows in flight stay in registers.
        // Row rr starts output row rr (of the segment), feeds rr - 1 and completes rr - 2.  The rows before the
        // first and after the last output row accumulate into registers that are re-initialised or dropped.
        auto step = [&](int rr, auto ph_tag) {
            constexpr int PH = decltype(ph_tag)::value;
            asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");      // row rr has landed
            __syncthreads();
            if (rr + kRing - 1 < nr) fill(rr + kRing - 1, wr);
            asm volatile("cp.async.commit_group;" ::: "memory");
            const T *row = reinterpret_cast<const T *>(sm + rd) + c0 * CH + 2 * pair, *rowx = reinterpret_cast<const T *>(sm + rd + kXOff) + c0 * CH + 2 * pair;
            wr = rd;                    // the row read now is the one refilled after the next barrier
            rd = rd + kSlot == kRing * kSlot ? 0 : rd + kSlot;
            float2 gv[kCols + 2];
#pragma unroll
            for (int v = 0; v < kCols + 2; ++v) gv[v] = load_pair(row + v * CH);
#pragma unroll
            for (int p = 0; p < kCols; ++p) {
                o[PH][p] = bs;
                if (BWD) xr[PH][p] = load_pair(rowx + p * CH);      // zero past the segment's last row and past the grid
            }
            if (BWD && rr >= 1 && rr < nr - 1) {                    // rows of the segment itself
#pragma unroll
                for (int p = 0; p < kCols; ++p) {
                    accb = add2(accb, gv[p + 1]);
                }
            }
#pragma unroll
            for (int u = 0; u < 3; ++u)
#pragma unroll
                for (int p = 0; p < kCols; ++p) {
                    float2 &a = o[(PH + 3 - u) % 3][p];
                    const float2 xx = xr[(PH + 3 - u) % 3][p];
#pragma unroll
                    for (int v = 0; v < 3; ++v) {
                        a = fma2(wf[u][v], gv[p + v], a);
                        if (BWD) acc[u][v] = fma2(xx, gv[p + v], acc[u][v]);
                    }
                }
            if (rr >= 2) {
#pragma unroll
                for (int p = 0; p < kCols; ++p)
                    if (p < ncol) store_pair(orow + (size_t)p * D, o[(PH + 1) % 3][p]);
                orow += row_elems;
            }
        };
        for (int rr = 0; rr < nr; rr += 3) {
            step(rr, std::integral_constant<int, 0>{});
            if (rr + 1 < nr) step(rr + 1, std::integral_constant<int, 1>{});
            if (rr + 2 < nr) step(rr + 2, std::integral_constant<int, 2>{});
        }
    }
    pdl_launch_dependents();
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (!BWD) return;
    __syncthreads();
    // partial[part][k][D]: k = stored tap index 0..8, 9 = bias
    float *red = reinterpret_cast<float *>(sm);
#pragma unroll
    for (int k = 0; k < 10; ++k)
        *reinterpret_cast<float2 *>(red + (grp * 10 + k) * CH + 2 * pair) = k < 9 ? acc[k / 3][k % 3] : accb;
    __syncthreads();
    for (int idx = threadIdx.x; idx < 10 * CH; idx += kConvThreads) {
        const int k = idx / CH, c = idx - k * CH;
        if (chb * CH + c >= D) continue;
        float sum = red[k * CH + c];
#pragma unroll
        for (int j = 1; j < kGroups; ++j) sum += red[(j * 10 + k) * CH + c];
        partial[((size_t)blockIdx.y * 10 + (k < 9 ? stored_tap(k / 3, k % 3, dir) : 9)) * D + chb * CH + c] = sum;
    }
}

// Sums of the CTA rows' partial sums: lanes hold neighbouring values (whole lines per load), warp s of the block
// adds every kSumWarps-th partial sum, then the warps' sums are added in order (fixed, whatever the scheduling).
// One warp per value, its lanes striding over the partial sums and each load a sector of its own: 6.3 us for 64
// partial sums of 11520 values, 3.2 us now.
constexpr int kSumWarps = 8;
__global__ void __launch_bounds__(32 * kSumWarps)
srem_dwconv_wgrad_sum(const float *__restrict__ partial, float *__restrict__ dw, float *__restrict__ dbias,
                      int nslab, int D)
{
    __shared__ float sh[kSumWarps][32];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, idx = blockIdx.x * 32 + lane;
    pdl_wait();
    pdl_launch_dependents();
    float sum = 0.f;
    if (idx < 10 * D) {
#pragma unroll 8
        for (int s = wp; s < nslab; s += kSumWarps) sum += partial[(size_t)s * 10 * D + idx];
    }
    sh[wp][lane] = sum;
    __syncthreads();
    if (wp != 0 || idx >= 10 * D) return;
#pragma unroll
    for (int s = 1; s < kSumWarps; ++s) sum += sh[s][lane];
    if (idx < 9 * D) dw[idx] = sum;
    else if (dbias != nullptr) dbias[idx - 9 * D] = sum;
}

// Rows of a strip cut evenly into at most one segment per 8 rows (two halo rows come on top): 9 rows become 5 + 4, and the
// last segment may be short (65 rows: eight of 8 and one of 1).
struct StripCut {
    int nseg, seg_rows;
    StripCut(int want, int gh)
    {
        nseg = want > (gh + 7) / 8 ? (gh + 7) / 8 : want;
        if (nseg < 1) nseg = 1;
        seg_rows = (gh + nseg - 1) / nseg;
        nseg = (gh + seg_rows - 1) / seg_rows;
    }
};

// What both directions take: the grid of the one-tile kernel, which serves small problems and bounds them all.
bool sizes_served(int B, int gh, int nchb) { return (gh + TY - 1) / TY <= 65535 && (size_t)B * nchb <= 65535; }

template <bool BWD>
dig_status launch_strip(const void *src, const void *w, const void *bias, void *dst, const void *x, float *partial, int B, int gh,
                        int gw, int D, int dir, int dtype, dim3 grid, StripCut cut, int nstrips, cudaStream_t stream)
{
    const int strips_x = (gw + TX - 1) / TX;
    auto go = [&](auto t, auto to) {
        using T = decltype(t);
        using TO = decltype(to);
        launch_pdl(srem_dwconv3x3_strip<T, TO, BWD>, grid, dim3(Cfg<T>::kThreads), 0, stream, (const T *)src, (const T *)w,
                   (const T *)bias, (TO *)dst, (const T *)x, partial, B, gh, gw, D, dir, strips_x, cut.nseg, cut.seg_rows, nstrips);
    };
    switch (dtype) {
        case DIG_F32: go(float{}, float{}); break;
        case DIG_BF16: go(__nv_bfloat16{}, __nv_bfloat16{}); break;
        case DIG_BF16_F32OUT: go(__nv_bfloat16{}, float{}); break;
        default: return DIG_ERR_INVALID_ARG;
    }
    return cuda_ok(cudaGetLastError());
}

}  // namespace

dig_status launch_dwconv(const void *x, const void *w, const void *bias, void *y, int B, int gh,
                         int gw, int D, int dir, int dtype, cudaStream_t stream)
{
    const int CH = dtype == DIG_F32 ? Cfg<float>::CH : Cfg<__nv_bfloat16>::CH;
    const int nchb = (D + CH - 1) / CH;
    const dim3 grid((gw + TX - 1) / TX, (gh + TY - 1) / TY, B * nchb);
    if (!sizes_served(B, gh, nchb)) return DIG_ERR_UNSUPPORTED;
    KernelTimer t(KID_DWCONV, stream);
    // grids with at least one tile per resident CTA: strips of TX columns walked row by row, cut into row
    // segments so that as many CTAs as stay resident have work
    const long long ntiles = (long long)grid.x * grid.y * grid.z;
    const int sms = device_sm_count();
    if (sms <= 0) return DIG_ERR_CUDA;
    const int resident = sms * kStripCtas;
    if (ntiles >= resident && ntiles < (1ll << 31)) {
        const long long cols = (long long)grid.x * B, want = resident / nchb;    // strips of a channel block before the cut
        const StripCut cut((int)(want / cols), gh);                 // one wave of CTAs where the strips allow it
        const long long nstrips = cols * cut.nseg;
        const dim3 pgrid(nchb, (unsigned)(want < 1 ? 1 : nstrips < want ? nstrips : want));
        return launch_strip<false>(x, w, bias, y, nullptr, nullptr, B, gh, gw, D, dir, dtype, pgrid, cut, (int)nstrips, stream);
    }
    switch (dtype) {
        case DIG_F32:
            launch_pdl(srem_dwconv3x3<float, float>, grid, dim3(Cfg<float>::kThreads), 0, stream,
                       (const float *)x, (const float *)w, (const float *)bias, (float *)y, gh, gw, D, nchb, dir);
            break;
        case DIG_BF16:
            launch_pdl(srem_dwconv3x3<__nv_bfloat16, __nv_bfloat16>, grid, dim3(Cfg<__nv_bfloat16>::kThreads), 0, stream,
                       (const __nv_bfloat16 *)x, (const __nv_bfloat16 *)w, (const __nv_bfloat16 *)bias,
                       (__nv_bfloat16 *)y, gh, gw, D, nchb, dir);
            break;
        case DIG_BF16_F32OUT:
            launch_pdl(srem_dwconv3x3<__nv_bfloat16, float>, grid, dim3(Cfg<__nv_bfloat16>::kThreads), 0, stream,
                       (const __nv_bfloat16 *)x, (const __nv_bfloat16 *)w, (const __nv_bfloat16 *)bias,
                       (float *)y, gh, gw, D, nchb, dir);
            break;
        default: return DIG_ERR_INVALID_ARG;
    }
    return cuda_ok(cudaGetLastError());
}

// CTA rows of the reverse mode, one partial sum each: no more than stay resident together, so that their strip loops end
// together, and no more than one per kWgPixels pixels (with one per 128, which the filter sums alone wanted, small grids
// had too few CTAs for dx: 11 x 5 x 8 pixels of 712 channels 11.0 us, 8 x 11 x 32 of 592 23.9, 6.6 and 11.8 now; 8 x 32 x 32 of 384 18.8 -> 13.9).
static long long slabs_for(int B, int gh, int gw, int nchb)
{
    int sms = device_sm_count();
    if (sms <= 0) sms = 148;            // sizing call without a device: the count the launch will most likely see
    const long long cap = sms * kStripCtas / nchb, n = ((long long)B * gh * gw + kWgPixels - 1) / kWgPixels;
    return n < cap ? n : cap > 0 ? cap : 1;
}

size_t dwconv_bwd_workspace_bytes(int B, int gh, int gw, int D)
{
    const int CH = Cfg<__nv_bfloat16>::CH;         // the wider block of the two storage types: the most CTA rows
    return (size_t)slabs_for(B, gh, gw, (D + CH - 1) / CH) * 10 * (size_t)D * sizeof(float);
}

dig_status launch_dwconv_bwd(const void *x, const void *w, const void *dy, void *dx, float *dw, float *dbias,
                             int B, int gh, int gw, int D, int dir, int dtype, float *partial, cudaStream_t stream)
{
    // Strips are cut into row segments until every CTA row has one.
    const int CHb = dtype == DIG_F32 ? Cfg<float>::CH : Cfg<__nv_bfloat16>::CH;
    const int nchb = (D + CHb - 1) / CHb;
    if (!sizes_served(B, gh, nchb)) return DIG_ERR_UNSUPPORTED;
    if (device_sm_count() <= 0) return DIG_ERR_CUDA;
    long long nslab = slabs_for(B, gh, gw, nchb);
    const int strips_x = (gw + TX - 1) / TX;
    const long long base = (long long)B * strips_x;
    const StripCut cut((int)(nslab / base), gh);                    // rounded down: no CTA row gets a second strip while others have one
    const long long nstrips = base * cut.nseg;
    if (nslab > nstrips) nslab = nstrips;
    if (nslab > 65535 || nstrips >= (1ll << 31)) return DIG_ERR_UNSUPPORTED;
    {
        KernelTimer t(KID_DWCONV_WGRAD, stream);
        const dig_status st = launch_strip<true>(dy, w, nullptr, dx, x, partial, B, gh, gw, D, dir, dtype, dim3(nchb, (unsigned)nslab), cut,
                                                 (int)nstrips, stream);
        if (st != DIG_OK) return st;
    }
    if (cudaGetLastError() != cudaSuccess) return DIG_ERR_CUDA;
    KernelTimer t(KID_DWCONV_WGRAD, stream);
    launch_pdl(srem_dwconv_wgrad_sum, dim3((10 * D + 31) / 32), dim3(32 * kSumWarps), 0, stream, (const float *)partial, dw, dbias,
               (int)nslab, D);
    return cuda_ok(cudaGetLastError());
}

}  // namespace dig
