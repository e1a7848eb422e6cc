// tcgen05 "sweep" kernels of chunkwise gated linear attention (Eq. attn_gla, Section 3.5): the
// recurrence S_t = diag(exp(a_t)) S_{t-1} + k_t^T v_t, o_t = q_t S_t worked in 64-token tiles, with
// the d_k x d_v state held on chip while a CTA walks over a segment of consecutive tiles.
//
// A sequence of N tiles is cut into segments of G tiles; one CTA sweeps one segment.
//   forward : sweep_local_fwd  per segment, from a zero state: the state it leaves and its total decay
//             seg_scan         per sequence, over the few segment ends: the state entering each segment
//             sweep_fwd        per segment, from its true entry state: out = tril(Qc Kc^T) V + Qc Sc per tile
//   backward: sweep_local_bwd  per segment, from a zero state: per (sub-)chunk the state entering it in fp16
//                              and the decay since the segment start; the segment's contribution to the
//                              state gradient
//             seg_scan         forward over the states, backward over the state gradients, gate-gradient carry
//             sweep_bwd        per segment in reverse: dq, dk, dv, dgate with the state gradient on chip
// Where the sequences are not cut (one segment each) the forward pass is sweep_fwd alone, started from the
// start state, and the backward pass without state arguments needs no scan: its local sweep only stores
// the per-chunk states, and the entry state, incoming gradient and carry of every segment are zero.
// Per (sub-)chunk, with Lam the cumulative gate inside it, c = Lam_end / 2 per channel,
//   Qc = q exp(Lam - c), Kc = k exp(c - Lam), Sc = diag(exp(c)) S_in, Dc = diag(exp(c)) D_out:
//   P   = tril(Qc Kc^T)                         dP = tril(dO V^T)
//   out = P V + Qc Sc                           S_out = exp(2c) S_in + exp(c) (Kc^T V)
//   dq  = (dP Kc + dO Sc^T) exp(Lam - c)        dk = (dP^T Qc + V Dc^T) exp(c - Lam)
//   dv  = P^T dO + Kc Dc                        D_in = exp(2c) D_out + exp(c) (Qc^T dO)
//   dgate_j = sum_{r >= j} (q dq - k dk)_r  (running over the whole sequence in reverse scan order)
// In the backward sweep S_in = S_local + diag(G) S_segment, G the decay since the segment start, so
// dO Sc^T = dO Sc_local^T + (dO S_segment^T) diag(exp(c) G): two products and one fused multiply-add.
//
// A tile whose gates sum to too much for one centring, or that was asked for in shorter chunks, is worked in sub-chunks.  Two
// of 32 rows share one pass through a kernel's phases: operands are built once, each row centred on its own half, scores are
// block-diagonal, and only what acts through the state or its gradient is done per half, the later half with the second
// group of products.  The results are those of two passes bit for bit.  48 sequences of 1961 tokens in chunks of 32, d = 72:
// the four kernels 42 + 56 + 76 + 108 us with a pass per half, 28 + 38 + 56 + 84 now; 48 of 4096, d = 64, half of the heads at
// tau = 4, where one tile in six is divided and the CTA with most of them is the last: 35 + 49 + 48 + 94, now 30 + 42 + 46 + 94 (the
// backward sweep shares a pass in chunks of 32 only).
//
// Every product is a tcgen05.mma (kind::f16, fp16 operands, fp32 accumulators in tensor memory) issued by
// one thread of the last warp, which otherwise works like the others: all threads build operand tiles, mask the
// scores and post-process accumulators, phase by phase (columns.cuh holds the work split).  Rows of the
// next tile are prefetched into registers; two CTAs of 256 threads share an SM, so one builds while the
// other's products are in the tensor pipe.
#include "columns.cuh"
#include "sweep.cuh"
#include "sweep_plan.cuh"

namespace dig {
namespace {

using namespace sw;

struct SweepArgs {
    const bf16 *q, *k, *v, *d_out;
    const float *gate;
    void *out, *dq, *dk, *dv;
    float *dgate;
    float *seg_state, *seg_gamma, *seg_dstate, *seg_carry;
    __half *seg_state16, *slot_s;
    float *slot_g;
    const float *s_in;      // forward pass with uncut sequences: the start state ([B*H][d][d], may be null) ...
    float *s_out;           // ... and where the final state goes (may be null)
    int *status;
    int accumulate;
    int scanned;            // backward pass: a segment scan ran (else every segment's entry state, gradient and carry are zero)
    Geom g;
    Plan plan;
    // Several scan orders in one forward launch: g.B = batch * orders sequences per head; order i (two bits each in dirs) reads
    // the same inputs and writes out_stride elements behind the one before.
    int batch;
    uint32_t dirs, out_stride;
};

// Batch entry, head, scan order and place of the results of sequence bh.  ORDERS: of several scan orders in one launch.
struct Seq {
    int b, h, dir;
    uint32_t oo;
};
template <bool ORDERS>
__device__ __forceinline__ Seq seq_of(const SweepArgs &a, int bh)
{
    Seq s{bh / a.g.H, 0, a.g.dir, 0u};
    s.h = bh - s.b * a.g.H;
    if (ORDERS) {
        const int i = s.b / a.batch;
        s.b -= i * a.batch;
        s.dir = (int)(a.dirs >> (2 * i)) & 3;
        s.oo = (uint32_t)i * a.out_stride;
    }
    return s;
}

// A condition known to the compiler, for code that also takes a bool.
template <bool B> struct Const {
    __device__ constexpr operator bool() const { return B; }
};

// Tiles of two 32-row sub-chunks (Halves).  The code that works both in one pass costs tiles that are not divided so.
//   Local sweeps and, in sweeps of more than kPlainTiles tiles, the forward sweep have it for chunks of 32 and more.  The forward
//   sweep of fewer tiles takes a pass each: its launches wait for instructions (one tile per CTA, 144 CTAs, d = 64: a forward
//   pass of 12.6 us against 13.0; four tiles, 768 CTAs: 46.2 and 46.9).
//   The backward sweep has it for chunks of 32 only (see there).
//   Chunks of 16, whose tiles are never divided so, have instances without any of it: 48 sequences of 12544 tokens, d = 64, local
//   sweeps 238 us forward and 303 backward with it, 233 and 280 without; 16 of 16384, d = 72, backward sweep 427 and 419.
constexpr int kPlainTiles = 4;

// ---- shared phases ------------------------------------------------------------------------------
__device__ __forceinline__ void cta_setup(Ctl *ctl, int nbar, uint32_t tmem_cols, char *tiles, int tile_bytes)
{
    const int tid = threadIdx.x;
    if (tid < 32) tmem_alloc(&ctl->tmem_base, tmem_cols);
    if (tid == 32) {
        for (int i = 0; i < nbar; ++i) mbar_init(&ctl->bar[i], 1);
        fence_barrier_init();
    }
    zero_smem(tiles, tile_bytes);
    fence_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
}
__device__ __forceinline__ void cta_teardown(Ctl *ctl, uint32_t tmem_cols)
{
    tc_fence_before_sync();
    __syncthreads();
    if (threadIdx.x < 32) tmem_dealloc(ctl->tmem_base, tmem_cols);
}

// Bounded wait whose verdict (with the thread's earlier ones) is uniform over the warp: tcgen05.ld must never
// run under a lane-divergent condition.
__device__ __forceinline__ bool wait_all(uint64_t *bar, uint32_t parity, int *status, bool ok)
{
    const bool done = mbar_wait(bar, parity, status);
    return __all_sync(0xffffffffu, done && ok) != 0;
}

#define SYNC_OR_DIE()                               \
    do {                                            \
        if (!__syncthreads_and(ok)) {               \
            ok = false;                             \
            goto die;                               \
        }                                           \
    } while (0)

// =================================================================================================
// sweep_local_fwd: the state a segment leaves from a zero start, and its total decay.  The tiles are walked from the
// segment's end, so the decay from a tile's centre to the end is known when its product is: the state is the plain
// sum of 2^(that decay) (Kc^T V), kept in tensor memory.  One barrier per tile or sub-chunk (two sub-chunks of 32 rows are
// one step with two products): behind it lie the group sums of this tile and the operand rows of the step before, whose
// product is issued there and added once this step's operands are built; operand tiles and sums have two buffers, and the
// rows of the next tile are loaded a whole tile ahead.
// Bound by the latency of its phases.  48 sequences of 4096 tokens, d = 64: 40 us with the state in registers, decayed
// once per tile in scan order, 30 us now; 16 of 16384, d = 72: 80 -> 52 us (63 with the sum in registers, which spills).
// One operand exponent for the whole way to the segment's end would let the matrix unit add the products up (29 and
// 43 us), but fp16 then loses what decays below 2^-25 even where nothing larger follows: errors of 0.3 of RMS where a
// segment's keys lie in its first tile.
// =================================================================================================
template <int D>
struct LocalFwdSmem {
    using C = Cfg<D>;
    using L = Col<D>;
    static constexpr int kBuf = 2 * C::TILE_T;                                // tK tV
    static constexpr int kPad = L::X ? 16 * C::CHT - C::TILE_T : 0;           // the corner's operand reads past its tile
    static constexpr size_t bytes = 2 * kBuf + kPad + 2 * 8 * D * 4 + 4 * T * 4 + sizeof(Ctl);
    static constexpr uint32_t aSum = 2 * L::ACCS;                             // accumulator columns: products of one pass (of two halves), the sum
    static constexpr uint32_t tmem_cols = 3 * L::ACCS <= 128 ? 128 : 256;
};

template <int D, bool ORDERS, Halves HALVES>
__global__ void __launch_bounds__(Col<D>::NT, 2)
sweep_local_fwd(const SweepArgs a)
{
    using C = Cfg<D>;
    using L = Col<D>;
    using SM = LocalFwdSmem<D>;
    extern __shared__ __align__(128) char smem[];
    float *sTot = reinterpret_cast<float *>(smem + 2 * SM::kBuf + SM::kPad);
    int *rowOff = reinterpret_cast<int *>(sTot + 2 * 8 * D);          // ring of four tiles
    Ctl *ctl = reinterpret_cast<Ctl *>(rowOff + 4 * T);

    const int tid = threadIdx.x;
    cta_setup(ctl, 1, SM::tmem_cols, smem, 2 * SM::kBuf + SM::kPad);
    const Who<D> w;
    const StateOf<D> sm(w);
    const uint32_t tmem = warp_uniform(ctl->tmem_base), tl = tmem + ((uint32_t)(32 * w.q4) << 16);
    const Geom &g = a.g;
    const Plan &pl = a.plan;
    Cols<D, false, false> raw;
    Cols<D, false, false> nxt;                          // rows and gates of the next tile, a whole tile ahead of their use
    bool ok = true, first = true;                       // first: nothing of this segment is in the sum
    uint32_t it = 0;                                    // operand tiles built so far: buffer it & 1, phase of their products' barrier it & 1
    const int total = g.B * g.H * pl.nseg;

    // products of the tiles built last (before the barrier just passed), one or one per half
    Weight w1{}, w2{};                                  // their weights
    bool pending = false, pair = false;
    auto issue_step = [&]() {
        if (w.issuer() && elect_one()) {
            char *tK = smem + ((it - 1) & 1) * SM::kBuf;
            tc_fence_after_sync();
            if (HALVES != kHalvesTogether || !pair) {
                issue_state<D>(tmem, tK, tK + C::TILE_T);
            } else {
                issue_state<D, kHighRows>(tmem, tK, tK + C::TILE_T);
                issue_state<D, kLowRows>(tmem + L::ACCS, tK, tK + C::TILE_T);
            }
            mma_commit(&ctl->bar[0]);
        }
    };
    auto add_step = [&](uint32_t parity) {
        ok = wait_all(&ctl->bar[0], parity, a.status, ok);
        tc_fence_after_sync();
        if (ok) {
            add_product<D>(tl + SM::aSum, tl, sm, w1, first);
            if (HALVES == kHalvesTogether && pair) add_product<D>(tl + SM::aSum, tl + L::ACCS, sm, w2, false);
        }
        first = false;
        tc_fence_before_sync();
    };

    pdl_wait();
    for (int sid = blockIdx.x; sid < total; sid += gridDim.x) {
        const int bh = sid / pl.nseg, sg = sid - bh * pl.nseg;
        const Seq sq = seq_of<ORDERS>(a, bh);
        const int t0 = sg * pl.G, t1 = min(t0 + pl.G, pl.ntile);
        first = true;
        RowSum after{0.f, 0.f};                                         // gates of the tiles behind
        pending = false;
        if (tid < 3 * T && t1 - 1 - (tid >> 6) >= t0) {
            const int tile = t1 - 1 - (tid >> 6);
            rowOff[(tile & 3) * T + (tid & 63)] = tile_row_offset(g, pl, sq.dir, sq.b, sq.h, D, tile, tid & 63);
        }
        __syncthreads();
        {
            uint32_t off[9];
            row_offsets<D>(rowOff + ((t1 - 1) & 3) * T, w, off);
            load_gates(raw.g, a.gate, off);
            load_rows(raw, a.q, a.k, a.v, a.d_out, off);
            if (t1 - 2 >= t0) {
                row_offsets<D>(rowOff + ((t1 - 2) & 3) * T, w, off);
                load_gates(nxt.g, a.gate, off);
            }
            const int nrow = g.L - (t1 - 1) * T;
            if (nrow < T) { clear_tail_rows(raw, w, nrow); clear_tail_gates(raw, w, nrow); }
            group_prefix<D>(raw, raw.g, w, sTot + ((t1 - 1) & 1) * 8 * D);
        }
        for (int tile = t1 - 1; tile >= t0; --tile) {
            const int nrow = min(T, g.L - tile * T);
            const float *tot = sTot + (tile & 1) * 8 * D;
            tc_fence_before_sync();
            SYNC_OR_DIE();                                             // group totals are there, the step before is built
            if (pending) issue_step();
            if (tid < T && tile - 3 >= t0) rowOff[((tile - 3) & 3) * T + tid] = tile_row_offset(g, pl, sq.dir, sq.b, sq.h, D, tile - 3, tid);
            if (tile > t0) {
                uint32_t ro[9];
                row_offsets<D>(rowOff + ((tile - 1) & 3) * T, w, ro);
                load_rows(nxt, a.q, a.k, a.v, a.d_out, ro);
            }
            Tot tt = tile_totals<D>(tot, w);
            const RowSum mine = row_sum<D>(sm, tt);
            const int s = divide_tile<D, HALVES>(tot, w, pl.sub_max, a.status, tt);
            centre_rows<D>(raw, w, centred(tt.before, tt.all), centred(tt.xbefore, tt.xall), nrow);
            const bool halves = HALVES == kHalvesTogether && s == T / 2 && nrow > T / 2;            // two sub-chunks at once, a product each
            const int step = halves ? T : s, nsub = (nrow + step - 1) / step;
            for (int u = nsub - 1; u >= 0; --u) {
                if (u < nsub - 1) {
                    tc_fence_before_sync();
                    SYNC_OR_DIE();
                    issue_step();
                }
                char *tK = smem + (it & 1) * SM::kBuf;                  // what read it last has been added
                build_rows<D>(raw, w, nullptr, tK, tK + C::TILE_T, nullptr, 8 * w.grp >= u * step && 8 * w.grp < (u + 1) * step);
                fence_async_smem();
                if (pending) add_step((it - 1) & 1);
                pending = true;
                pair = halves;
                ++it;
                // gates from the centre to the segment's end
                if (halves) {
                    const RowSum low = row_sum<D>(sm, half_totals<D, 0>(tot, w)), high = row_sum<D>(sm, half_totals<D, 1>(tot, w));
                    w1 = weight_of<D>(high, after);
                    w2 = weight_of<D>(low, after + high);
                } else if (s < T) {
                    w1 = weight_of<D>(row_sum<D>(sm, window_totals<D>(tot, w, u * s / 8, (u + 1) * s / 8)),
                                      after + row_sum<D>(sm, window_totals<D>(tot, w, (u + 1) * s / 8, 8)));
                } else {
                    w1 = weight_of<D>(mine, after);
                }
            }
            after = after + mine;
            if (tile > t0) {
                group_prefix<D>(raw, nxt.g, w, sTot + ((tile - 1) & 1) * 8 * D);       // only the last tile of a sequence has a tail
                if (tile - 2 >= t0) {
                    uint32_t ro[9];
                    row_offsets<D>(rowOff + ((tile - 2) & 3) * T, w, ro);
                    load_gates(nxt.g, a.gate, ro);
                    prefetch_rows<D, false, false>(a.q, a.k, a.v, a.d_out, rowOff + ((tile - 2) & 3) * T, w);
                }
#pragma unroll
                for (int j = 0; j < raw.N; ++j) {
                    raw.k[j] = nxt.k[j];
                    raw.v[j] = nxt.v[j];
                }
            }
        }
        tc_fence_before_sync();
        SYNC_OR_DIE();
        issue_step();
        add_step((it - 1) & 1);
        if (ok) acc_to_global<D>(tl + SM::aSum, sm, a.seg_state + (size_t)sid * D * D);
        tc_fence_before_sync();
        put_row_sums<D>(a.seg_gamma + (size_t)sid * D, w, sm, after);
    }
die:
    cta_teardown(ctl, SM::tmem_cols);
    pdl_launch_dependents();
}

// =================================================================================================
// sweep_local_bwd: what the backward sweep needs of a segment from a zero state.  In scan order, the state
// in registers: per (sub-)chunk the state entering it (scaled to its centre, fp16) and the decay since the
// segment start.  GRAD: also the segment's contribution to the gradient of the state entering it, the sum of
// 2^(gates from the segment start to the centre) (Qc^T dO), in tensor memory (the state and the rows take the
// registers).  A backward pass over uncut sequences needs only the states.
// Pipelined over the (sub-)chunks: the products of one run while the next one's operand tiles are built (two
// buffers of tiles and accumulators), and are folded into the sums one step later.  48 sequences of 4096 tokens, d = 64:
// 60 us with both sums in registers and no pipelining, 45 us now; 16 of 16384, d = 72: 122 -> 101 us.
// =================================================================================================
template <int D, bool GRAD>
struct LocalBwdSmem {
    using C = Cfg<D>;
    using L = Col<D>;
    static constexpr int kBuf = (GRAD ? 4 : 2) * C::TILE_T;                   // (tQ) tK tV (tG)
    static constexpr int kPad = L::X ? 16 * C::CHT - C::TILE_T : 0;           // the corner's operand reads past its tile
    static constexpr size_t bytes = 2 * kBuf + kPad + 2 * 8 * D * 4 + 4 * T * 4 + sizeof(Ctl);
    // accumulator columns: two of the state's products, two of the gradient's, the gradient's sum
    static constexpr uint32_t aW = 2 * L::ACCS, aSum = 4 * L::ACCS;
    static constexpr uint32_t cols = (GRAD ? 5 : 2) * L::ACCS;
    static constexpr uint32_t tmem_cols = cols <= 64 ? 64 : cols <= 128 ? 128 : 256;
    static_assert(cols <= 256, "tensor memory of two CTAs");
};

template <int D, bool GRAD, Halves HALVES>
__global__ void __launch_bounds__(Col<D>::NT, 2)
sweep_local_bwd(const SweepArgs a)
{
    using C = Cfg<D>;
    using L = Col<D>;
    using SM = LocalBwdSmem<D, GRAD>;
    extern __shared__ __align__(128) char smem[];
    float *sTot = reinterpret_cast<float *>(smem + 2 * SM::kBuf + SM::kPad);
    int *rowOff = reinterpret_cast<int *>(sTot + 2 * 8 * D);          // ring of four tiles
    Ctl *ctl = reinterpret_cast<Ctl *>(rowOff + 4 * T);

    const int tid = threadIdx.x;
    cta_setup(ctl, 2, SM::tmem_cols, smem, 2 * SM::kBuf + SM::kPad);
    const Who<D> w;
    const StateOf<D> sm(w);
    const uint32_t tmem = warp_uniform(ctl->tmem_base), tl = tmem + ((uint32_t)(32 * w.q4) << 16);
    const Geom &g = a.g;
    const Plan &pl = a.plan;
    float S[L::NPS][8];
    Cols<D, GRAD, GRAD> raw;
    bool ok = true;
    uint32_t it = 0;                                    // (sub-)chunks worked so far: accumulators it & 1, their barrier's phase (it >> 1) & 1
    uint32_t nbuf = 0;                                  // operand tiles built so far: buffer nbuf & 1
    const int total = g.B * g.H * pl.nseg;

    auto load_tile = [&](int tile) {
        uint32_t off[9];
        row_offsets<D>(rowOff + (tile & 3) * T, w, off);
        load_gates(raw.g, a.gate, off);
        load_rows(raw, a.q, a.k, a.v, a.d_out, off);
    };
    // S <- 2^2c S + 2^c (Kc^T V), sum <- sum + 2^(.) (Qc^T dO): the products of step i
    Decay dec;
    Weight wt{};
    bool pending = false, first = true;                 // the step before waits to be folded; nothing of this segment is in the sum
    auto fold = [&](uint32_t i) {
        ok = wait_all(&ctl->bar[i & 1], (i >> 1) & 1, a.status, ok);
        tc_fence_after_sync();
        if (ok) {
            fold_state<D>(tl + (i & 1) * L::ACCS, sm, S, dec);
            if (GRAD) add_product<D>(tl + SM::aSum, tl + SM::aW + (i & 1) * L::ACCS, sm, wt, first);
        }
        first = false;
        tc_fence_before_sync();
    };

    pdl_wait();
    for (int sid = blockIdx.x; sid < total; sid += gridDim.x) {
        const int bh = sid / pl.nseg, sg = sid - bh * pl.nseg, b = bh / g.H, h = bh - b * g.H;
        const int t0 = sg * pl.G, t1 = min(t0 + pl.G, pl.ntile);
        get_state<D>(nullptr, sm, S);
        RowSum since{0.f, 0.f};                                         // gates since the segment start
        pending = false;
        first = true;
        if (tid < 2 * T) rowOff[((t0 + (tid >> 6)) & 3) * T + (tid & 63)] = tile_row_offset(g, pl, g.dir, b, h, D, t0 + (tid >> 6), tid & 63);
        __syncthreads();
        load_tile(t0);
        {
            const int nrow = g.L - t0 * T;
            if (nrow < T) { clear_tail_rows(raw, w, nrow); clear_tail_gates(raw, w, nrow); }
            group_prefix<D>(raw, raw.g, w, sTot + (t0 & 1) * 8 * D);
        }
        for (int tile = t0; tile < t1; ++tile) {
            const int nrow = min(T, g.L - tile * T);
            const bool more = tile + 1 < t1;
            float *tot = sTot + (tile & 1) * 8 * D;
            SYNC_OR_DIE();                                             // group totals are there
            if (tid < T && tile + 2 < t1) rowOff[((tile + 2) & 3) * T + tid] = tile_row_offset(g, pl, g.dir, b, h, D, tile + 2, tid);
            Tot tt = tile_totals<D>(tot, w);
            const RowSum mine = row_sum<D>(sm, tt);
            const int s = divide_tile<D, HALVES>(tot, w, pl.sub_max, a.status, tt);
            centre_rows<D>(raw, w, centred(tt.before, tt.all), centred(tt.xbefore, tt.xall), nrow);
            // Two sub-chunks of 32 rows: one pass, a product each in either accumulator, the state between them as soon as the
            // first is done (nothing of them stays for the next pass).
            const bool halves = HALVES == kHalvesTogether && s == T / 2 && nrow > T / 2;
            const int step = halves ? T : s, nsub = (nrow + step - 1) / step, nslot = halves ? 2 : nsub;
            for (int u = 0; u < nsub; ++u, ++it, ++nbuf) {
                const int lo = u * step;
                const bool last = u == nsub - 1, on = 8 * w.grp >= lo && 8 * w.grp < lo + step;
                char *buf = smem + (nbuf & 1) * SM::kBuf;
                char *tQ = buf, *tK = GRAD ? tQ + C::TILE_T : buf, *tV = tK + C::TILE_T, *tG = tV + C::TILE_T;
                build_rows<D>(raw, w, tQ, tK, tV, tG, on);
                RowSum own, before = since;                            // gates of the sub-chunk and before it
                if (halves) {
                    own = row_sum<D>(sm, half_totals<D, 0>(tot, w));
                } else if (s < T) {
                    before = since + row_sum<D>(sm, window_totals<D>(tot, w, 0, lo / 8));
                    own = row_sum<D>(sm, window_totals<D>(tot, w, lo / 8, (lo + s) / 8));
                } else {
                    own = mine;
                }
                const Decay now = decay_of<D>(own);
                Weight wnow{};
                if (GRAD) wnow = weight_of<D>(own, before);
                size_t slot = ((size_t)(nslot - 1 - u) * g.B * g.H + bh) * pl.ntile + tile;
                put_row_sums<D>(a.slot_g + slot * D, w, sm, before);
                const bool late = L::X && halves;                      // registers: rows after the second half's state
                if (last && more && !late) load_tile(tile + 1);
                if (halves && pending) {                               // both accumulators have to be free
                    fold(it - 1);
                    pending = false;
                }
                fence_async_smem();
                tc_fence_before_sync();
                __syncthreads();
                if (w.issuer() && elect_one()) {
                    tc_fence_after_sync();
                    const uint32_t x = (it & 1) * L::ACCS, y = L::ACCS - x;
                    if (!halves) {
                        issue_state<D>(tmem + x, tK, tV);                                          // Kc^T V
                        if (GRAD) issue_state<D>(tmem + SM::aW + x, tQ, tG);                       // Qc^T dO
                        mma_commit(&ctl->bar[it & 1]);
                    } else {
                        issue_state<D, kLowRows>(tmem + x, tK, tV);
                        if (GRAD) issue_state<D, kLowRows>(tmem + SM::aW + x, tQ, tG);
                        mma_commit(&ctl->bar[it & 1]);
                        issue_state<D, kHighRows>(tmem + y, tK, tV);
                        if (GRAD) issue_state<D, kHighRows>(tmem + SM::aW + y, tQ, tG);
                        mma_commit(&ctl->bar[(it + 1) & 1]);
                    }
                }
                // the register prefetch alone does not cover the memory latency of tiles this short
                if (last && tile + 2 < t1) prefetch_rows<D, GRAD, GRAD>(a.q, a.k, a.v, a.d_out, rowOff + ((tile + 2) & 3) * T, w);
                if (last && tile + 2 < t1) prefetch_gates<D>(a.gate, rowOff + ((tile + 2) & 3) * T, w);
                if (pending) fold(it - 1);
                dec = now;
                wt = wnow;
                put_state<D, D * 16>(reinterpret_cast<char *>(a.slot_s + slot * (D * D)), sm, S, dec);
                pending = true;
                if (halves) {
                    fold(it++);
                    before = since + own;
                    own = row_sum<D>(sm, half_totals<D, 1>(tot, w));
                    slot -= (size_t)g.B * g.H * pl.ntile;
                    put_row_sums<D>(a.slot_g + slot * D, w, sm, before);
                    dec = decay_of<D>(own);
                    if (GRAD) wt = weight_of<D>(own, before);
                    put_state<D, D * 16>(reinterpret_cast<char *>(a.slot_s + slot * (D * D)), sm, S, dec);
                    if (late && more) load_tile(tile + 1);
                }
            }
            since = since + mine;
            if (more) {                                                // the next tile's gate sums while the products run
                const int nr = g.L - (tile + 1) * T;
                if (nr < T) { clear_tail_rows(raw, w, nr); clear_tail_gates(raw, w, nr); }
                group_prefix<D>(raw, raw.g, w, sTot + ((tile + 1) & 1) * 8 * D);
            }
        }
        fold(it - 1);
        save_state<D>(a.seg_state + (size_t)sid * D * D, sm, S);
        if (GRAD && ok) acc_to_global<D>(tl + SM::aSum, sm, a.seg_dstate + (size_t)sid * D * D);
        put_row_sums<D>(a.seg_gamma + (size_t)sid * D, w, sm, since);
        tc_fence_before_sync();
    }
die:
    cta_teardown(ctl, SM::tmem_cols);
    pdl_launch_dependents();
}

// =================================================================================================
// seg_scan: the recurrence over segment ends, 16 lanes per (sequence, state row), a lane four neighbouring
// value channels (and four more at d = 72, lanes 0 and 1).  Forward: seg_state[s] (state a segment
// leaves from a zero start) becomes the state entering segment s.  Backward flavour: seg_dstate[s] (the
// segment's own contribution) becomes the gradient with respect to the state leaving segment s, seg_carry
// the gate-gradient carried into the segment from later ones, seg_state16 an fp16 copy of the entry states
// in the dense chunk-major order the backward sweep bulk-copies.
// Bound by the latency of its loads, which do not depend on the recurrence: NF (NB on the way back) segments are in
// flight together.  Few segments get a kernel of their own with short loops, since fetching the instructions of the long
// ones takes longer than they do (6 segments x 48 sequences, d = 64: 5.2 us in the long kernel, 3.6 in the short
// one; backward flavour 9.1 and 5.6).  49 segments x 6 sequences, d = 64: 8.0 us with 8 lanes per row and fewer loads in
// flight, 6.1 with 16 lanes, 5.5 us now; backward flavour, 18 x 16, d = 72: 14.6 -> 10.1 -> 7.9 us.  A whole warp
// per row: 12.9 us (five shuffles per row, half of the lanes idle in the second piece).
// =================================================================================================
constexpr int kScanRows = 8;                          // state rows per block
constexpr int kScanFew = 8;                           // segments up to which the short kernel serves
template <int D, bool BWD, bool MANY>
__global__ void __launch_bounds__(16 * kScanRows)
seg_scan(float *seg_state, const float *seg_gamma, float *seg_dstate, float *seg_carry, __half *seg_state16,
         const float *s_in, float *s_out, const float *ds_out, float *ds_in, int nseg)
{
    constexpr int NV = (D / 4 + 15) / 16;             // float4 pieces per lane
    // segments whose loads are in flight together, on the way forward and on the way back
    constexpr int NF = MANY ? (NV == 1 ? 32 : 18) : (NV == 1 ? 8 : 6), NB = MANY ? (NV == 1 ? 16 : 9) : NF;
    const int bh = blockIdx.x, c = blockIdx.y * kScanRows + (threadIdx.x >> 4), lane = threadIdx.x & 15;
    static_assert(D % kScanRows == 0, "whole blocks of rows");
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const size_t dd = (size_t)D * D, io = bh * dd + (size_t)c * D + 4 * lane, st0 = (size_t)bh * nseg * dd + (size_t)c * D + 4 * lane;
    const float *gam0 = seg_gamma + (size_t)bh * nseg * D + c;
    auto has = [&](int i) { return i == 0 || lane < D / 4 - 16; };
    auto ld = [&](const float *p, int i) { return has(i) ? *reinterpret_cast<const float4 *>(p + 64 * i) : zero; };
    auto st = [&](float *p, int i, float4 v) { if (has(i)) *reinterpret_cast<float4 *>(p + 64 * i) = v; };
    auto step = [](float g, float4 x, float4 t) { return make_float4(g * x.x + t.x, g * x.y + t.y, g * x.z + t.z, g * x.w + t.w); };
    pdl_wait();
    pdl_launch_dependents();
    float4 s[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) s[i] = s_in ? ld(s_in + io, i) : zero;
    for (int sg0 = 0; sg0 < nseg; sg0 += NF) {
        float4 t[NF][NV];
        float gam[NF];
#pragma unroll
        for (int j = 0; j < NF; ++j) {
            const int sg = sg0 + j;
            if (sg < nseg) {
                gam[j] = gam0[(size_t)sg * D];
#pragma unroll
                for (int i = 0; i < NV; ++i) t[j][i] = ld(seg_state + st0 + sg * dd, i);
            }
        }
#pragma unroll
        for (int j = 0; j < NF; ++j) {
            const int sg = sg0 + j;
            if (sg < nseg) {
                const float gm = exp2f(gam[j]);
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    st(seg_state + st0 + sg * dd, i, s[i]);
                    if (BWD && has(i)) {
                        const int e = 4 * lane + 64 * i;
                        const __half2 h[2] = {__floats2half2_rn(s[i].x, s[i].y), __floats2half2_rn(s[i].z, s[i].w)};
                        char *dst = reinterpret_cast<char *>(seg_state16 + ((size_t)bh * nseg + sg) * dd);
                        *reinterpret_cast<uint2 *>(dst + ((e >> 3) * D + c) * 16 + (e & 7) * 2) = *reinterpret_cast<const uint2 *>(h);
                    }
                    s[i] = step(gm, s[i], t[j][i]);
                }
            }
        }
    }
    if (s_out) {
#pragma unroll
        for (int i = 0; i < NV; ++i) st(s_out + io, i, s[i]);
    }
    if (BWD) {
        float4 d[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) d[i] = ds_out ? ld(ds_out + io, i) : zero;
        // s holds the state leaving the last segment; walking back, it is replaced by the entry state of
        // the segment just handled, which is the state leaving the one before it
        for (int sg0 = nseg - 1; sg0 >= 0; sg0 -= NB) {
            float4 t[NB][NV], sp[NB][NV];
            float gam[NB];
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const int sg = sg0 - j;
                if (sg >= 0) {
                    gam[j] = gam0[(size_t)sg * D];
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        t[j][i] = ld(seg_dstate + st0 + sg * dd, i);
                        sp[j][i] = ld(seg_state + st0 + sg * dd, i);
                    }
                }
            }
            float dot[NB];
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const int sg = sg0 - j;
                dot[j] = 0.f;
                if (sg >= 0) {
                    const float gm = exp2f(gam[j]);
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        st(seg_dstate + st0 + sg * dd, i, d[i]);
                        dot[j] += s[i].x * d[i].x + s[i].y * d[i].y + s[i].z * d[i].z + s[i].w * d[i].w;
                        d[i] = step(gm, d[i], t[j][i]);
                        s[i] = sp[j][i];
                    }
                }
            }
#pragma unroll
            for (int m = 8; m >= 1; m >>= 1)
#pragma unroll
                for (int j = 0; j < NB; ++j) dot[j] += __shfl_xor_sync(0xffffffffu, dot[j], m);
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (lane == j && sg0 - j >= 0) seg_carry[((size_t)bh * nseg + sg0 - j) * D + c] = dot[j];
        }
        if (ds_in) {
#pragma unroll
            for (int i = 0; i < NV; ++i) st(ds_in + io, i, d[i]);
        }
    }
}

// =================================================================================================
// sweep_fwd: a segment from its entry state; writes out.
// Bound by the latency of its phases (three barriers and two waits for products per tile; IPC 1.5, two CTAs per
// SM).  16 sequences of 16384 tokens, d = 72: 114 us with the row-chunk work split, 76 us now; 768 of 256, d = 64
// (uncut): 60 -> 48 us; 48 of 4096: 62 -> 51.  Three CTAs per SM on 80 registers spill: 72 us there.
// =================================================================================================
template <int D, typename TO>
struct FwdSmem {
    using C = Cfg<D>;
    using L = Col<D>;
    static constexpr int kTiles = 3 * C::TILE_T + C::TILE_S + C::TILE_P;      // tQ tK tV tS tP
    static constexpr size_t bytes = kTiles + Staging<D, TO>::kBytes + 8 * D * 4 + 4 * T * 4 + sizeof(Ctl);
    static constexpr uint32_t aP = 0, aO = 32, aU = aO + L::HW;               // accumulator columns
    static constexpr uint32_t tmem_cols = 128;
    static_assert(aU + L::ACCS <= tmem_cols, "tensor memory");
};

template <int D, typename TO, Halves HALVES>
__global__ void __launch_bounds__(Col<D>::NT, 2)
sweep_fwd(const SweepArgs a)
{
    using C = Cfg<D>;
    using L = Col<D>;
    using SM = FwdSmem<D, TO>;
    constexpr bool ORDERS = sizeof(TO) == 4;            // sums over scan orders have fp32 results
    extern __shared__ __align__(128) char smem[];
    char *tQ = smem, *tK = tQ + C::TILE_T, *tV = tK + C::TILE_T, *tS = tV + C::TILE_T, *tP = tS + C::TILE_S;
    char *stage = smem + SM::kTiles;
    float *sTot = reinterpret_cast<float *>(stage + Staging<D, TO>::kBytes);
    int *rowOff = reinterpret_cast<int *>(sTot + 8 * D);               // ring of four tiles: the one before, this one, the next
    Ctl *ctl = reinterpret_cast<Ctl *>(rowOff + 4 * T);

    const int tid = threadIdx.x;
    cta_setup(ctl, 1, SM::tmem_cols, smem, SM::kTiles);
    const Who<D> w;
    const StateOf<D> sm(w);
    const uint32_t tmem = warp_uniform(ctl->tmem_base), tl = tmem + ((uint32_t)(32 * w.q4) << 16);
    const Geom &g = a.g;
    const Plan &pl = a.plan;
    float S[L::NPS][8];
    Cols<D, true, false> raw;
    bool ok = true;
    int cur = 0, staged = 0;                            // rows of the tile before that wait in the staging buffer
    const int total = g.B * g.H * pl.nseg;
    TO *out = reinterpret_cast<TO *>(a.out);

    auto load_tile = [&](int slot) {
        uint32_t off[9];
        row_offsets<D>(rowOff + slot * T, w, off);
        load_gates(raw.g, a.gate, off);
        load_rows(raw, a.q, a.k, a.v, nullptr, off);
    };
    // The first tile's rows are inputs of the call: their loads need not wait for the scan kernel (whose own
    // wait covered whatever produced them).  Uncut sequences have no kernel in front that has waited: wait first.
    auto prime = [&](int sid) {
        const int bh = sid / pl.nseg, sg = sid - bh * pl.nseg;
        const Seq sq = seq_of<ORDERS>(a, bh);
        if (tid < T) rowOff[cur * T + tid] = tile_row_offset(g, pl, sq.dir, sq.b, sq.h, D, sg * pl.G, tid);
        __syncthreads();
        load_tile(cur);
    };
    if (pl.nseg == 1) pdl_wait();
    if ((int)blockIdx.x < total) prime(blockIdx.x);
    pdl_wait();
    for (int sid = blockIdx.x; sid < total; sid += gridDim.x) {
        const int bh = sid / pl.nseg, sg = sid - bh * pl.nseg;
        const Seq sq = seq_of<ORDERS>(a, bh);
        const int t0 = sg * pl.G, t1 = min(t0 + pl.G, pl.ntile);
        if (pl.nseg == 1) get_state<D>(a.s_in ? a.s_in + (size_t)sid * D * D : nullptr, sm, S);      // uncut: no scan ran
        else get_state<D>(a.seg_state + (size_t)sid * D * D, sm, S);
        if (sid != (int)blockIdx.x) prime(sid);
        {
            const int nrow = g.L - t0 * T;
            if (nrow < T) { clear_tail_rows(raw, w, nrow); clear_tail_gates(raw, w, nrow); }
            group_prefix<D>(raw, raw.g, w, sTot);
        }
        for (int tile = t0; tile < t1; ++tile) {
            const int nrow = min(T, g.L - tile * T), nxt = (cur + 1) & 3, prv = (cur + 3) & 3;
            const bool more = tile + 1 < t1;
            tc_fence_before_sync();
            SYNC_OR_DIE();                                       // group totals are there, the previous tile's products are done
            if (tid < T && more) rowOff[nxt * T + tid] = tile_row_offset(g, pl, sq.dir, sq.b, sq.h, D, tile + 1, tid);
            // Where some channel's gates sum to too much for one centring (or shorter chunks were asked for) the tile
            // is worked in sub-chunks with their own centring.  Two of 32 rows share one pass through the phases below
            // (`halves`): both are built and scored at once, the state between them is formed after the scores and read by the
            // upper half's rows alone.  Shorter ones take a pass each, the other rows of the operand tiles zero.
            const Tot whole = tile_totals<D>(sTot, w);
            Tot tt = whole;
            const int s = divide_tile<D, HALVES, HALVES == kHalvesApart>(sTot, w, pl.sub_max, a.status, tt);
            centre_rows<D>(raw, w, centred(tt.before, tt.all), centred(tt.xbefore, tt.xall), nrow);
            // At d = 64 the two kinds of pass are compiled apart (768 sequences of 256 tokens 49.2 us without halves, 50.9
            // with the branches, 50.0 so); at d = 72 registers would spill.
            auto passes = [&](auto kind) {
                const bool halves = kind;
                const int step = halves ? T : s, nsub = halves ? 1 : (nrow + step - 1) / step;
                for (int u = 0; u < nsub; ++u) {
                    const int lo = u * step, hi = lo + step;
                    const bool last = u == nsub - 1;
                    build_rows<D>(raw, w, tQ, tK, tV, nullptr, 8 * w.grp >= lo && 8 * w.grp < hi);
                    Tot tu = whole;
                    if (halves) tu = half_totals<D, 0>(sTot, w);
                    else if (s < T) tu = window_totals<D>(sTot, w, lo / 8, hi / 8);
                    Decay dec = decay_of<D>(row_sum<D>(sm, tu));
                    put_state<D, C::CHS>(tS, sm, S, dec);            // Sc = diag(2^c) S
                    fence_async_smem();
                    tc_fence_before_sync();
                    __syncthreads();
                    if (w.issuer() && elect_one()) {
                        tc_fence_after_sync();
                        issue_scores<D>(tmem + SM::aP, tQ, tK);                                       // Qc Kc^T
                        if (!halves) mma_commit(&ctl->bar[0]);
                        issue_split<D, C::KS, C::CHS>(tmem + SM::aO, tQ, tS, false);                  // Qc Sc
                        if (!halves) {
                            issue_state<D>(tmem + SM::aU, tK, tV);                                    // Kc^T V
                        } else {
                            issue_state<D, kLowRows>(tmem + SM::aU, tK, tV);
                            mma_commit(&ctl->bar[0]);
                        }
                    }
                    if (staged) flush_rows<D>(out, sq.oo, stage, rowOff + prv * T, w, staged, a.accumulate != 0);
                    staged = 0;
                    if (last && more) load_tile(nxt);
                    ok = wait_all(&ctl->bar[0], 0, a.status, ok);          // completes twice per iteration: parities 0, 1
                    tc_fence_after_sync();
                    if (halves && ok) {                                    // the state between the halves
                        fold_state<D>(tl + SM::aU, sm, S, dec);
                        tu = half_totals<D, 1>(sTot, w);
                        dec = decay_of<D>(row_sum<D>(sm, tu));
                        put_state<D, C::CHS>(tS, sm, S, dec);
                    }
                    // Scores of row r16: lanes 0-15 hold the even 8-token chunks, lanes 16-31 the odd ones.  Keep s <= t, the
                    // diagonal has weight 1.  Chunks above the diagonal of all 16 rows of the warp are never written (the tile
                    // starts out zero), pairs below it need no selects.
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int pr = w.cg + 2 * i;
                        if (ok && pr <= w.q4) {                // uniform over the warp
                            float p[8];
                            tmem_ld8(tl + SM::aP + 8 * pr, p);
                            const int sc = 2 * pr + w.hf;
                            if (pr == w.q4) {
#pragma unroll
                                for (int e = 0; e < 8; ++e) p[e] = (8 * sc + e <= w.r16) ? p[e] : 0.f;
                            } else if (halves && pr < 2 && w.q4 >= 2) {        // the lower half acts on the upper one through the state
#pragma unroll
                                for (int e = 0; e < 8; ++e) p[e] = 0.f;
                            }
                            *reinterpret_cast<uint4 *>(tP + sc * C::CHT + w.r16 * 16) = pack_h8(p);
                        }
                    }
                    fence_async_smem();
                    tc_fence_before_sync();
                    __syncthreads();
                    if (w.issuer() && elect_one()) {
                        tc_fence_after_sync();
                        if (halves) {
                            issue_split<D, C::KS, C::CHS, kHighRows>(tmem + SM::aO, tQ, tS, false);
                            issue_state<D, kHighRows>(tmem + SM::aU, tK, tV);
                        }
                        if (HALVES == kHalvesTogether) issue_weighted<D>(tmem + SM::aO, tP, tV);                          // + P V
                        else issue_split<D, T / 16, C::CHT>(tmem + SM::aO, tP, tV, true);
                        mma_commit(&ctl->bar[0]);
                    }
                    if (last && more) {                                // the next tile's gate sums while the products run
                        const int nr = g.L - (tile + 1) * T;
                        if (nr < T) { clear_tail_rows(raw, w, nr); clear_tail_gates(raw, w, nr); }
                        group_prefix<D>(raw, raw.g, w, sTot);
                    }
                    ok = wait_all(&ctl->bar[0], 1, a.status, ok);
                    tc_fence_after_sync();
                    if (ok) {
                        const bool inrow = w.r16 >= lo && w.r16 < min(hi, nrow);
#pragma unroll
                        for (int i = 0; i < L::NPO; ++i) {
                            const int jc = w.cg + 2 * i;
                            if (jc < L::NV0) {                        // uniform over the warp
                                float o[8];
                                tmem_ld8(tl + SM::aO + 8 * jc, o);
                                if (inrow && jc < (w.hf ? L::NV1 : L::NV0)) stage_row<D, TO>(stage, w.r16, (w.hf ? L::NV0 : 0) + jc, o);
                            }
                        }
                        fold_state<D>(tl + SM::aU, sm, S, dec);
                    }
                    if (!last) {                              // the operand tiles and the accumulators are free again
                        tc_fence_before_sync();
                        if (!__syncthreads_and(ok)) return false;
                    }
                }
                return true;
            };
            [[maybe_unused]] const bool two = s == T / 2 && nrow > T / 2;
            bool done;
            if constexpr (HALVES != kHalvesTogether) done = passes(Const<false>{});
            else if constexpr (L::X) done = passes(two);
            else done = two ? passes(Const<true>{}) : passes(Const<false>{});
            if (!done) {
                ok = false;
                goto die;
            }
            staged = nrow;
            cur = nxt;
        }
        SYNC_OR_DIE();
        flush_rows<D>(out, sq.oo, stage, rowOff + ((cur + 3) & 3) * T, w, staged, a.accumulate != 0);
        staged = 0;
        if (pl.nseg == 1 && a.s_out) save_state<D>(a.s_out + (size_t)sid * D * D, sm, S);
    }
die:
    cta_teardown(ctl, SM::tmem_cols);
    pdl_launch_dependents();
}

// =================================================================================================
// sweep_bwd: a segment in reverse scan order with the state gradient on chip.
// After the second group of products the dq and dk accumulators go through shared memory (over the
// operand tiles that are spent by then) to the column threads, which still hold the decay exponents of
// their rows: they scale and store dq and dk, form q dq - k dk and sum it down their rows.
// Two sub-chunks of 32 rows in one pass only for chunks of 32: the code for it slows whole tiles down by 4% at d = 64 (92.4 -> 96 us
// on 768 sequences of 256 tokens) and 2.5% at d = 72, also compiled apart per tile (101 us, spills) or per CTA (98.7; short launches
// then wait for instructions: 25.4 -> 34 us on 48 sequences of 1024).  Heads of low gate temperature in chunks of 32 pay for it: tiles
// in sub-chunks of 16 or 8 rows (tau = 2) take 5% longer than without that code.
// Bound by latency like the forward sweep.  48 sequences of 4096 tokens, d = 64: 140 us with the row-chunk work
// split, 94 us now; 16 of 16384, d = 72: 252 -> 181 us.
// =================================================================================================
template <int D, typename TO>
struct BwdSmem {
    using C = Cfg<D>;
    using L = Col<D>;
    static constexpr int LDP = D + 4;                                          // floats per row of an accumulator buffer
    static constexpr int kBuf = T * LDP * 4;
    static constexpr int kOver = 2 * C::TILE_T + C::TILE_S;                    // tV tG tD: spent when the accumulators are complete
    static constexpr int kRegion = 2 * kBuf > kOver ? 2 * kBuf : kOver;
    static constexpr int kTiles = 2 * C::TILE_T + kRegion + 2 * C::TILE_P + 2 * C::TILE_S;      // tQ tK | tV tG tD .. | tP tdP | tS tI
    // dv leaves through a staging buffer (see Staging): one of its own at d = 64; at d = 72, where two CTAs leave no
    // room for it, the zero-start state's tile, whose refill then waits for the copy; fp32 results do not fit there
    // and are stored directly
    static constexpr bool kStage = D == 64 || sizeof(TO) == 2, kOwnStage = D == 64;
    static constexpr int kStageBytes = kOwnStage ? Staging<D, TO>::kBytes : 0;
    static_assert(!kStage || kOwnStage || Staging<D, TO>::kBytes <= C::NCH * C::CHS, "the state tile's zero chunk stays clean");
    static constexpr size_t bytes = kTiles + kStageBytes + (2 * 8 * D + 2 * D) * 4 + 2 * T * 4 + sizeof(Ctl);
    static constexpr uint32_t aP = 0, aQK = 64, aV = aQK + D, aW = aV + D;     // accumulator columns
    static constexpr uint32_t tmem_cols = 256;
    static_assert(aW + L::ACCS <= tmem_cols, "tensor memory");
};

__device__ __forceinline__ void store_pair(float *p, float x, float y, bool add)
{
    if (add) asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" :: "l"(p), "f"(x), "f"(y) : "memory");
    else *reinterpret_cast<float2 *>(p) = make_float2(x, y);
}
__device__ __forceinline__ void store_pair(bf16 *p, float x, float y, bool) { *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(x, y); }

template <int D, typename TO, Halves HALVES>
__global__ void __launch_bounds__(Col<D>::NT, 2)
sweep_bwd(const SweepArgs a)
{
    using C = Cfg<D>;
    using L = Col<D>;
    using SM = BwdSmem<D, TO>;
    extern __shared__ __align__(128) char smem[];
    char *tQ = smem, *tK = tQ + C::TILE_T, *tV = tK + C::TILE_T, *tG = tV + C::TILE_T, *tD = tG + C::TILE_T;
    char *tP = tV + SM::kRegion, *tdP = tP + C::TILE_P, *tS = tdP + C::TILE_P, *tI = tS + C::TILE_S;
    float *bufQ = reinterpret_cast<float *>(tV), *bufK = bufQ + T * SM::LDP;
    char *stage = SM::kOwnStage ? smem + SM::kTiles : tS;
    float *sTot = reinterpret_cast<float *>(smem + SM::kTiles + SM::kStageBytes), *sX = sTot + 8 * D, *sAux = sX + 8 * D;
    int *rowOff = reinterpret_cast<int *>(sAux + 2 * D);
    Ctl *ctl = reinterpret_cast<Ctl *>(rowOff + 2 * T);

    const int tid = threadIdx.x;
    cta_setup(ctl, 2, SM::tmem_cols, smem, SM::kTiles);
    const Who<D> w;
    const StateOf<D> sm(w);
    const uint32_t tmem = warp_uniform(ctl->tmem_base), tl = tmem + ((uint32_t)(32 * w.q4) << 16);
    uint64_t *barG1 = &ctl->bar[0], *barS = &ctl->bar[1];
    const Geom &g = a.g;
    const Plan &pl = a.plan;
    float Dst[L::NPS][8];
    Cols<D, true, true> raw;
    uint32_t par = 0;
    bool ok = true;
    int cur = 0;
    const int total = g.B * g.H * pl.nseg;
    TO *dq = reinterpret_cast<TO *>(a.dq), *dk = reinterpret_cast<TO *>(a.dk), *dv = reinterpret_cast<TO *>(a.dv);
    const bool acc_out = a.accumulate != 0, entry = a.scanned != 0;

    auto load_all = [&](int slot) {
        uint32_t off[9];
        row_offsets<D>(rowOff + slot * T, w, off);
        load_gates(raw.g, a.gate, off);
        load_rows(raw, a.q, a.k, a.v, a.d_out, off);
    };
    // The zero-start state of the (sub-)chunk worked after sub-chunk u of `tile` (whose slot is given): the issuing
    // thread asks for it once the tile of the one before is free.
    auto fetch_next = [&](int bh, size_t slot, int u, int tile, bool more) {
        if (w.issuer() && (u > 0 || more) && elect_one()) {
            const size_t nslot = u > 0 ? slot + (size_t)g.B * g.H * pl.ntile : (size_t)bh * pl.ntile + (tile - 1);
            const char *src = reinterpret_cast<const char *>(a.slot_s + nslot * (D * D));
            mbar_arrive_expect_tx(barS, (uint32_t)C::NCH * D * 16u);
            for (int j = 0; j < C::NCH; ++j) bulk_g2s(tS + j * C::CHS, src + j * D * 16, D * 16, barS);
        }
    };
    // the first tile's rows are inputs of the call: their loads need not wait for the scan kernel
    auto prime = [&](int sid) {
        const int bh = sid / pl.nseg, sg = sid - bh * pl.nseg;
        const Seq sq = seq_of<false>(a, bh);
        const int t1 = min(sg * pl.G + pl.G, pl.ntile);
        if (tid < T) rowOff[cur * T + tid] = tile_row_offset(g, pl, sq.dir, sq.b, sq.h, D, t1 - 1, tid);
        __syncthreads();
        load_all(cur);
    };
    if ((int)blockIdx.x < total) prime(blockIdx.x);
    pdl_wait();
    for (int sid = blockIdx.x; sid < total; sid += gridDim.x) {
        const int bh = sid / pl.nseg, sg = sid - bh * pl.nseg;
        const Seq sq = seq_of<false>(a, bh);
        const int t0 = sg * pl.G, t1 = min(t0 + pl.G, pl.ntile);
        // without a scan (uncut sequences, no state arguments) the entry state, the incoming state gradient and the carry are zero
        get_state<D>(entry ? a.seg_dstate + (size_t)sid * D * D : nullptr, sm, Dst);
        float2 carry = make_float2(0.f, 0.f), xcarry = carry;            // gate gradient carried in from later tiles
        if (entry) {
            carry = *reinterpret_cast<const float2 *>(a.seg_carry + (size_t)sid * D + w.c2);
            if (L::X) xcarry = *reinterpret_cast<const float2 *>(a.seg_carry + (size_t)sid * D + w.xc2);
        }
        if (sid != (int)blockIdx.x) prime(sid);
        if (w.issuer() && elect_one()) {
            // the zero-start state of the sub-chunk worked first (always slot 0 of its tile) and, once per
            // segment, the state entering the segment; later sub-chunks' states are fetched as soon as the
            // products of the one before are done
            const char *src = reinterpret_cast<const char *>(a.slot_s + ((size_t)bh * pl.ntile + (t1 - 1)) * (D * D));
            const char *seg16 = reinterpret_cast<const char *>(a.seg_state16 + (size_t)sid * D * D);
            mbar_arrive_expect_tx(barS, (entry ? 2u : 1u) * C::NCH * D * 16u);
            for (int j = 0; j < C::NCH; ++j) {
                bulk_g2s(tS + j * C::CHS, src + j * D * 16, D * 16, barS);
                if (entry) bulk_g2s(tI + j * C::CHS, seg16 + j * D * 16, D * 16, barS);
            }
        }
        {
            const int nrow = g.L - (t1 - 1) * T;
            if (nrow < T) { clear_tail_rows(raw, w, nrow); clear_tail_gates(raw, w, nrow); }
            group_prefix<D>(raw, raw.g, w, sTot);
        }
        for (int tile = t1 - 1; tile >= t0; --tile) {
            const int nrow = min(T, g.L - tile * T), nxt = cur ^ 1;
            const bool more = tile > t0;
            SYNC_OR_DIE();                                       // group totals are there, the accumulator buffers are free
            if (tid < T && more) rowOff[nxt * T + tid] = tile_row_offset(g, pl, sq.dir, sq.b, sq.h, D, tile - 1, tid);
            const Tot whole = tile_totals<D>(sTot, w);
            Tot tt = whole;
            const int s = divide_tile<D, HALVES>(sTot, w, pl.sub_max, a.status, tt);
            centre_rows<D>(raw, w, centred(tt.before, tt.all), centred(tt.xbefore, tt.xall), nrow);
            // Two sub-chunks of 32 rows share one pass: both are built, scored and finished at once; the upper half's products
            // with the gradient and the states come with the scores, the lower half's with the second group of products, once
            // the gradient between the halves is known.
            const bool halves = HALVES == kHalvesTogether && s == T / 2 && nrow > T / 2;
            const int step = halves ? T : s, nsub = (nrow + step - 1) / step;
            float2 tot = make_float2(0.f, 0.f), xtot = tot;      // sums of q dq - k dk over the group
            for (int u = nsub - 1; u >= 0; --u) {
                const int lo = u * step, hi = lo + step;
                const bool mine = 8 * w.grp >= lo && 8 * w.grp < hi;
                const size_t slot = ((size_t)(nsub - 1 - u) * g.B * g.H + bh) * pl.ntile + tile;
                build_rows<D>(raw, w, tQ, tK, tV, tG, mine);
                Tot tu = whole;
                if (halves) tu = half_totals<D, 1>(sTot, w);
                else if (s < T) tu = window_totals<D>(sTot, w, lo / 8, hi / 8);
                Decay dec = decay_of<D>(row_sum<D>(sm, tu));
                put_state<D, C::CHS>(tD, sm, Dst, dec);          // Dc = diag(2^c) D
                if (L::X) clear_pads<D>(tV, tG, tD);
                fence_async_smem();
                tc_fence_before_sync();
                __syncthreads();
                if (w.issuer() && elect_one()) {
                    ok = mbar_wait(barS, par, a.status) && ok;         // the state tiles have landed
                    tc_fence_after_sync();
                    const uint32_t sQ = smem_u32(tQ), sK = smem_u32(tK), sV = smem_u32(tV), sG = smem_u32(tG);
                    const uint32_t sS = smem_u32(tS), sI = smem_u32(tI), sD = smem_u32(tD);
                    issue<64, 64, false, false, C::KS, C::CHT, C::CHT>(tmem + SM::aP, sQ, sK, false);                   // Qc Kc^T
                    issue<64, 64, false, false, C::KS, C::CHT, C::CHT>(tmem + SM::aP + kHiLanes, sG, sV, false);        // dO V^T
                    if (!halves) mma_commit(barG1);
                    issue<64, D, false, false, C::KS, C::CHT, C::CHS>(tmem + SM::aQK, sG, sS, false);                   // dO Sc_local^T
                    if (entry) issue<64, D, false, false, C::KS, C::CHT, C::CHS>(tmem + SM::aV, sG, sI, false);         // dO S_segment^T
                    issue<64, D, false, false, C::KS, C::CHT, C::CHS>(tmem + SM::aQK + kHiLanes, sV, sD, false);        // V Dc^T
                    issue<64, D, false, true, C::KS, C::CHT, C::CHS>(tmem + SM::aV + kHiLanes, sK, sD, false);          // Kc Dc
                    if (!halves) {
                        issue_state<D>(tmem + SM::aW, tQ, tG);                                                          // Qc^T dO
                    } else {
                        issue_state<D, kHighRows>(tmem + SM::aW, tQ, tG);
                        mma_commit(barG1);
                    }
                }
                // decay from the segment start to a sub-chunk's centre; the lower half's in the second row of sAux
                auto put_aux = [&](float *aux, size_t sl, const Tot &t) {
                    const float2 G = *reinterpret_cast<const float2 *>(a.slot_g + sl * D + w.c2);
                    *reinterpret_cast<float2 *>(aux + w.c2) = make_float2(ex2(0.5f * t.all.x + G.x), ex2(0.5f * t.all.y + G.y));
                    if (L::X && w.xrow == 0) {
                        const float2 X = *reinterpret_cast<const float2 *>(a.slot_g + sl * D + w.xc2);
                        *reinterpret_cast<float2 *>(aux + w.xc2) = make_float2(ex2(0.5f * t.xall.x + X.x), ex2(0.5f * t.xall.y + X.y));
                    }
                };
                if (entry && w.grp == 0) {
                    put_aux(sAux, slot, tu);
                    if (halves) put_aux(sAux + D, slot + (size_t)g.B * g.H * pl.ntile, half_totals<D, 0>(sTot, w));
                }
                if (u == 0 && more) {
                    prefetch_gates<D>(a.gate, rowOff + nxt * T, w);
                    if (!kRowsEarly<D>) prefetch_rows<D, true, true>(a.q, a.k, a.v, a.d_out, rowOff + nxt * T, w);
                }
                if (kRowsEarly<D> && u == 0 && more) {
                    uint32_t ro[9];
                    row_offsets<D>(rowOff + nxt * T, w, ro);
                    load_rows(raw, a.q, a.k, a.v, a.d_out, ro);
                }
                ok = wait_all(barG1, 0, a.status, ok);         // completes twice per iteration: parities 0, 1
                tc_fence_after_sync();
                if (halves && ok) {
                    fetch_next(bh, slot, 1, tile, more);         // the lower half's state
                    fold_state<D>(tl + SM::aW, sm, Dst, dec);
                    tu = half_totals<D, 0>(sTot, w);
                    dec = decay_of<D>(row_sum<D>(sm, tu));
                    put_state<D, C::CHS>(tD, sm, Dst, dec);
                    par ^= 1;
                }
                // lanes 0-15: scores, lanes 16-31: dO V^T; keep s <= t, the diagonal has weight 1.  Column chunks
                // entirely above the diagonal for all rows of the warp are never written (the tiles start out zero),
                // chunks entirely below it need no selects.
                if (ok) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int sc = w.cg + 2 * i;
                        if (i <= w.q4) {                         // uniform over the warp: sc <= 2 q4 + 1
                            float p[8];
                            tmem_ld8(tl + SM::aP + 8 * sc, p);
                            if (i == w.q4) {
#pragma unroll
                                for (int e = 0; e < 8; ++e) p[e] = (8 * sc + e <= w.r16) ? p[e] : 0.f;
                            } else if (halves && i < 2 && w.q4 >= 2) {       // the halves meet through the states only
#pragma unroll
                                for (int e = 0; e < 8; ++e) p[e] = 0.f;
                            }
                            *reinterpret_cast<uint4 *>((w.hf ? tdP : tP) + sc * C::CHT + w.r16 * 16) = pack_h8(p);
                        }
                    }
                }
                fence_async_smem();
                tc_fence_before_sync();
                __syncthreads();
                if (w.issuer() && elect_one()) {
                    tc_fence_after_sync();
                    const uint32_t sQ = smem_u32(tQ), sK = smem_u32(tK), sG = smem_u32(tG);
                    const uint32_t sP = smem_u32(tP), sdP = smem_u32(tdP);
                    if (halves) {
                        const uint32_t sV = smem_u32(tV), sD = smem_u32(tD);
                        issue<64, D, false, false, C::KS, C::CHT, C::CHS, 128, kLowRows>(tmem + SM::aQK + kHiLanes, sV, sD, false);
                        issue<64, D, false, true, C::KS, C::CHT, C::CHS, 128, kLowRows>(tmem + SM::aV + kHiLanes, sK, sD, false);
                        issue_state<D, kLowRows>(tmem + SM::aW, tQ, tG);
                    }
                    if (halves) {
                        ok = mbar_wait(barS, par, a.status) && ok;
                        issue<64, D, false, false, C::KS, C::CHT, C::CHS, 128, kLowRows>(tmem + SM::aQK, sG, smem_u32(tS), false);
                    }
                    if (HALVES == kHalvesTogether) {
                        issue_triangle<D, false, C::CHT, C::CHT>(tmem + SM::aQK, sdP, sK);                              // + dP Kc
                        issue_triangle<D, true, C::CHT, C::CHT>(tmem + SM::aQK + kHiLanes, sdP, sQ);                    // + dP^T Qc
                        issue_triangle<D, true, C::CHT, C::CHT>(tmem + SM::aV + kHiLanes, sP, sG);                      // + P^T dO
                    } else {
                        issue<64, D, false, true, T / 16, C::CHT, C::CHT>(tmem + SM::aQK, sdP, sK, true);
                        issue<64, D, true, true, T / 16, C::CHT, C::CHT>(tmem + SM::aQK + kHiLanes, sdP, sQ, true);
                        issue<64, D, true, true, T / 16, C::CHT, C::CHT>(tmem + SM::aV + kHiLanes, sP, sG, true);
                    }
                    mma_commit(barG1);
                }
                ok = wait_all(barG1, 1, a.status, ok);
                tc_fence_after_sync();
                if (ok) {
                    if (SM::kOwnStage || !SM::kStage) fetch_next(bh, slot, u, tile, more);           // every product has completed
                    const bool inrow = w.r16 >= lo && w.r16 < min(hi, nrow);
                    float *buf = (w.hf ? bufK : bufQ) + w.r16 * SM::LDP;
#pragma unroll
                    for (int i = 0; i < (C::NCH + 1) / 2; ++i) {
                        const int jc = w.cg + 2 * i;
                        if (jc < C::NCH) {                       // uniform over the warp
                            // lanes 0-15: dq accumulator and dO S_segment^T; lanes 16-31: dk and dv accumulators
                            float x0[8], x1[8];
                            tmem_ld8_pair(tl + SM::aQK + 8 * jc, tl + SM::aV + 8 * jc, x0, x1);
                            if (w.hf) {
                                if (inrow) {
                                    if constexpr (SM::kStage) stage_row<D, TO>(stage, w.r16, jc, x1);
                                    else store_out8(dv + (uint32_t)rowOff[cur * T + w.r16] + 8 * jc, x1, acc_out);
                                }
                            } else if (entry) {
                                float hh[8];
                                ld8((halves && w.q4 < 2 ? sAux + D : sAux) + 8 * jc, hh);
#pragma unroll
                                for (int e = 0; e < 8; ++e) x0[e] = fmaf(hh[e], x1[e], x0[e]);
                            }
                            st8(buf + 8 * jc, x0);
                        }
                    }
                    fold_state<D>(tl + SM::aW, sm, Dst, dec);    // D <- 2^(2c) D + 2^c (Qc^T dO)
                }
                if (!kRowsEarly<D> && u == 0 && more) {
                    uint32_t ro[9];
                    row_offsets<D>(rowOff + nxt * T, w, ro);
                    load_rows(raw, a.q, a.k, a.v, a.d_out, ro);
                }
                tc_fence_before_sync();
                __syncthreads();
                if (mine) {                                      // uniform over the warp
                    // q dq = Qc (dq accumulator), k dk = Kc (dk accumulator): the decay factors cancel.  raw.g becomes
                    // the suffix sums of the group's rows.
                    const int *ro = rowOff + cur * T;
#pragma unroll
                    for (int j = raw.N - 1; j >= 0; --j) {
                        const int row = item_row(w, j), c2 = j < 8 ? w.c2 : w.xc2, o = pair_offset<D>(row, c2);
                        const float2 aq = *reinterpret_cast<const float2 *>(bufQ + row * SM::LDP + c2);
                        const float2 ak = *reinterpret_cast<const float2 *>(bufK + row * SM::LDP + c2);
                        const float2 q2 = __half22float2(*reinterpret_cast<const __half2 *>(tQ + o));
                        const float2 k2 = __half22float2(*reinterpret_cast<const __half2 *>(tK + o));
                        const float ex = raw.g[j].x, ey = raw.g[j].y;
                        const int r = ro[row];
                        if (row < nrow) {
                            store_pair(dq + (uint32_t)(r + c2), aq.x * ex2(ex), aq.y * ex2(ey), acc_out);
                            store_pair(dk + (uint32_t)(r + c2), ak.x * ex2(-ex), ak.y * ex2(-ey), acc_out);
                        }
                        const float x = q2.x * aq.x - k2.x * ak.x, y = q2.y * aq.y - k2.y * ak.y;
                        if (j < 8) {
                            tot.x += x;
                            tot.y += y;
                            raw.g[j] = tot;
                        } else {
                            xtot = make_float2(x, y);
#pragma unroll
                            for (int k = 1; k < 8; k <<= 1) {
                                const float px = __shfl_down_sync(0xffffffffu, xtot.x, 4 * k), py = __shfl_down_sync(0xffffffffu, xtot.y, 4 * k);
                                if (w.xrow + k < 8) { xtot.x += px; xtot.y += py; }
                            }
                            raw.g[j] = xtot;
                        }
                    }
                }
                // the state tile as staging holds this sub-chunk's rows only
                if (SM::kStage && (!SM::kOwnStage || u == 0)) flush_rows<D>(dv, 0u, stage, rowOff + cur * T, w, SM::kOwnStage || mine ? nrow : 0, acc_out);
                if (u > 0) {
                    fence_async_smem();
                    __syncthreads();                             // the accumulator buffers become operand tiles again
                    if (SM::kStage && !SM::kOwnStage) fetch_next(bh, slot, u, tile, more);
                }
                par ^= 1;
            }
            // gate gradient of the tile: suffix sums of q dq - k dk down the rows plus what later tiles carry in
            *reinterpret_cast<float2 *>(sX + w.grp * D + w.c2) = tot;
            if (L::X && w.xrow == 0) *reinterpret_cast<float2 *>(sX + w.grp * D + w.xc2) = xtot;
            if (SM::kStage && !SM::kOwnStage) fence_async_smem();
            __syncthreads();
            if (SM::kStage && !SM::kOwnStage) fetch_next(bh, 0, 0, tile, more);
            {
                const Tot after = later_totals<D>(sX, w);
                const float2 add = make_float2(carry.x + after.before.x, carry.y + after.before.y);
                const float2 xadd = make_float2(xcarry.x + after.xbefore.x, xcarry.y + after.xbefore.y);
                carry.x += after.all.x; carry.y += after.all.y;
                xcarry.x += after.xall.x; xcarry.y += after.xall.y;
                const int *ro = rowOff + cur * T;
#pragma unroll
                for (int j = 0; j < raw.N; ++j) {
                    const int r = ro[item_row(w, j)], c2 = j < 8 ? w.c2 : w.xc2;
                    if (item_row(w, j) < nrow) store_pair(a.dgate + (uint32_t)(r + c2), raw.g[j].x + (j < 8 ? add.x : xadd.x), raw.g[j].y + (j < 8 ? add.y : xadd.y), acc_out);
                }
            }
            if (more) {
                uint32_t ro[9];
                row_offsets<D>(rowOff + nxt * T, w, ro);
                load_gates(raw.g, a.gate, ro);
                group_prefix<D>(raw, raw.g, w, sTot);                   // only the last tile of a sequence has a tail, and it comes first
            }
            cur = nxt;
        }
    }
die:
    if (!ok && w.issuer() && elect_one()) mbar_wait(barS, par, a.status);      // let bulk copies in flight land
    cta_teardown(ctl, SM::tmem_cols);
    pdl_launch_dependents();
}

#undef SYNC_OR_DIE

// ---- host side ----------------------------------------------------------------------------------
template <typename K>
dig_status set_smem(K kern, size_t bytes)
{
    return ensure_dynamic_smem(reinterpret_cast<const void *>(kern), bytes);
}

// n scan orders (two bits each in dirs) of the same inputs; results of order i stand i * stride elements behind the first's.
template <int D, bool BWD>
dig_status run(const GlaArgs &ga, int n, uint32_t dirs, size_t stride)
{
    Geom g = ga.g;
    g.B *= n;
    const int sms = device_sm_count();
    int *status = device_status_ptr();
    if (!status || sms <= 0) return DIG_ERR_CUDA;
    const Plan pl = make_plan(g, sms, kPerSm, BWD);
    const SweepWs w = carve(reinterpret_cast<char *>(ga.ws), g, pl, BWD);
    if (w.bytes > ga.ws_bytes) return DIG_ERR_WORKSPACE;
    const long long total = (long long)g.B * g.H * pl.nseg;
    if (total > (1ll << 30) || (long long)g.B * g.L * g.H * D >= (1ll << 31)) return DIG_ERR_UNSUPPORTED;     // 31-bit row offsets
    SweepArgs a{};
    a.q = (const bf16 *)ga.q; a.k = (const bf16 *)ga.k; a.v = (const bf16 *)ga.v; a.d_out = (const bf16 *)ga.d_out;
    a.gate = ga.gate;
    a.out = ga.out; a.dq = ga.dq; a.dk = ga.dk; a.dv = ga.dv; a.dgate = ga.dgate;
    a.seg_state = w.seg_state; a.seg_gamma = w.seg_gamma; a.seg_dstate = w.seg_dstate; a.seg_carry = w.seg_carry;
    a.seg_state16 = w.seg_state16; a.slot_s = w.slot_s; a.slot_g = w.slot_g;
    a.status = status;
    a.accumulate = ga.accumulate;
    a.batch = ga.g.B;
    a.dirs = dirs;
    a.out_stride = (uint32_t)stride;
    a.g = g;
    a.plan = pl;
    const dim3 grid((unsigned)(total < (long long)sms * kPerSm ? total : (long long)sms * kPerSm)), block(Col<D>::NT);
    a.s_in = ga.sio.s_in;
    a.s_out = ga.sio.s_out;
    const bool sweep_only = !BWD && pl.nseg == 1;      // uncut sequences: the forward sweep starts from the start state itself
    const bool none = pl.sub_max < T / 2;                // chunks of 16: no tile is divided in two
    dig_status st;
    // backward pass over uncut sequences whose start-state gradient is not asked for: the segment's own
    // contribution to the state gradient is never used, the local sweep only has to store the states
    const bool states_only = BWD && pl.nseg == 1 && ga.sio.ds_in == nullptr;
    // ... and without state arguments there is nothing to scan: entry state, incoming gradient and carry are zero
    const bool scan = !sweep_only && !(states_only && ga.sio.s_in == nullptr && ga.sio.ds_out == nullptr);
    a.scanned = scan;
    if (!sweep_only) {
        void (*kern)(SweepArgs) = nullptr;
        size_t smem = 0;
        if constexpr (BWD) {
            kern = states_only ? (none ? sweep_local_bwd<D, false, kNoHalves> : sweep_local_bwd<D, false, kHalvesTogether>)
                               : (none ? sweep_local_bwd<D, true, kNoHalves> : sweep_local_bwd<D, true, kHalvesTogether>);
            smem = states_only ? LocalBwdSmem<D, false>::bytes : LocalBwdSmem<D, true>::bytes;
        } else {
            kern = n > 1 ? (none ? sweep_local_fwd<D, true, kNoHalves> : sweep_local_fwd<D, true, kHalvesTogether>)
                         : (none ? sweep_local_fwd<D, false, kNoHalves> : sweep_local_fwd<D, false, kHalvesTogether>);
            smem = LocalFwdSmem<D>::bytes;
        }
        if ((st = set_smem(kern, smem)) != DIG_OK) return st;
        KernelTimer t(KID_SW_LOCAL, ga.stream);
        launch_pdl(kern, grid, block, smem, ga.stream, a);
        if ((st = cuda_ok(cudaGetLastError())) != DIG_OK) return st;
    }
    if (scan) {
        auto kern = pl.nseg > kScanFew ? seg_scan<D, BWD, true> : seg_scan<D, BWD, false>;
        KernelTimer t(KID_SW_SCAN, ga.stream);
        launch_pdl(kern, dim3(g.B * g.H, D / kScanRows), dim3(16 * kScanRows), 0, ga.stream, w.seg_state, (const float *)w.seg_gamma, w.seg_dstate,
                   w.seg_carry, w.seg_state16, ga.sio.s_in, ga.sio.s_out, ga.sio.ds_out, ga.sio.ds_in, pl.nseg);
        if ((st = cuda_ok(cudaGetLastError())) != DIG_OK) return st;
    }
    const bool f32 = ga.dtype == DIG_BF16_F32OUT;
    if constexpr (!BWD) {
        constexpr size_t smem16 = FwdSmem<D, bf16>::bytes, smem32 = FwdSmem<D, float>::bytes;
        const bool two = pl.sub_max == T / 2 || pl.G > kPlainTiles;
        auto k16 = none ? sweep_fwd<D, bf16, kNoHalves> : two ? sweep_fwd<D, bf16, kHalvesTogether> : sweep_fwd<D, bf16, kHalvesApart>;
        auto k32 = none ? sweep_fwd<D, float, kNoHalves> : two ? sweep_fwd<D, float, kHalvesTogether> : sweep_fwd<D, float, kHalvesApart>;
        if ((st = set_smem(k16, smem16)) != DIG_OK || (st = set_smem(k32, smem32)) != DIG_OK) return st;
        KernelTimer t(KID_SW_FWD, ga.stream);
        launch_pdl(f32 ? k32 : k16, grid, block, f32 ? smem32 : smem16, ga.stream, a);
    } else {
        constexpr size_t smem16 = BwdSmem<D, bf16>::bytes, smem32 = BwdSmem<D, float>::bytes;
        const bool two = pl.sub_max == T / 2;
        auto k16 = none ? sweep_bwd<D, bf16, kNoHalves> : two ? sweep_bwd<D, bf16, kHalvesTogether> : sweep_bwd<D, bf16, kHalvesApart>;
        auto k32 = none ? sweep_bwd<D, float, kNoHalves> : two ? sweep_bwd<D, float, kHalvesTogether> : sweep_bwd<D, float, kHalvesApart>;
        if ((st = set_smem(k16, smem16)) != DIG_OK || (st = set_smem(k32, smem32)) != DIG_OK) return st;
        KernelTimer t(KID_SW_BWD, ga.stream);
        launch_pdl(f32 ? k32 : k16, grid, block, f32 ? smem32 : smem16, ga.stream, a);
    }
    return cuda_ok(cudaGetLastError());
}

}  // namespace

bool sweep_supports(int dk, int dv, int chunk, int dtype)
{
    if (dtype != DIG_BF16 && dtype != DIG_BF16_F32OUT) return false;
    (void)chunk;                     // every chunk size is worked in 64-token tiles, shorter ones as sub-chunks
    return dk == dv && (dk == 64 || dk == 72);
}

// SMs for sizes, which can be asked for without a device.
static int device_sms()
{
    const int sms = device_sm_count();
    return sms > 0 ? sms : 148;
}

size_t sweep_workspace_bytes(const Geom &g, bool backward)
{
    return launch_bytes(g, device_sms(), backward, 1);
}

namespace {

dig_status sweep_orders(const GlaArgs &a, bool backward, int n, uint32_t dirs, size_t stride)
{
    if (backward) return a.g.dk == 64 ? run<64, true>(a, n, dirs, stride) : run<72, true>(a, n, dirs, stride);
    return a.g.dk == 64 ? run<64, false>(a, n, dirs, stride) : run<72, false>(a, n, dirs, stride);
}

// Sums over n buffers of fp32 results, in order, to the caller's tensors (fp32, or rounded to the nearest even bf16), 8
// elements per thread; blockIdx.y selects the tensor.
struct SumArgs {
    const float *src[4];
    void *dst[4];
    bool f32[4];
};
__global__ void __launch_bounds__(256) sum_orders(const SumArgs a, int n, size_t stride, size_t n8)
{
    pdl_wait();
    pdl_launch_dependents();
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n8) return;
    const float *src = a.src[blockIdx.y] + 8 * i;
    float f[4][8];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (k < n) ld8(src + k * stride, f[k]);
#pragma unroll
    for (int k = 1; k < 4; ++k)
        if (k < n)
#pragma unroll
            for (int e = 0; e < 8; ++e) f[0][e] += f[k][e];
    if (a.f32[blockIdx.y]) store_out8(static_cast<float *>(a.dst[blockIdx.y]) + 8 * i, f[0]);
    else store_out8(static_cast<bf16 *>(a.dst[blockIdx.y]) + 8 * i, f[0]);
}

}  // namespace

// Several scan orders summed (Algorithm 2 / Algorithm 3): groups of orders one after the other, each launch adding
// its fp32 results to the same buffers, which are summed and rounded to the storage type once at the end.  An element of a
// buffer gets one addition per launch and the launches follow one another on the stream, so the sum does not depend on
// scheduling.
size_t sweep_multi_workspace_bytes(const Geom &g, bool backward, int dtype)
{
    const SumPlans plans(g, device_sms(), backward, dtype);
    size_t most = 0;
    for (int n = 1; n <= 4; ++n) {
        const size_t b = plans.of(n, SIZE_MAX).bytes();
        most = b > most ? b : most;
    }
    return most;
}

namespace {

dig_status sweep_multi(const GlaArgs &a0, bool backward, unsigned mask)
{
    GlaArgs a = a0;
    const size_t elems = (size_t)a.g.B * a.g.L * a.g.H * a.g.dk;          // d_k = d_v
    const int n = __builtin_popcount(mask);
    const SumPlan plan = SumPlans(a.g, device_sms(), backward, a0.dtype).of(n, a0.ws_bytes);
    if (plan.bytes() > a0.ws_bytes) return DIG_ERR_WORKSPACE;
    const int k = plan.k;
    char *buffers = reinterpret_cast<char *>(a0.ws);
    a.ws = reinterpret_cast<float *>(buffers + plan.buffer * plan.buffers);
    a.ws_bytes = plan.launch;
    void *const result[4] = {backward ? a0.dq : a0.out, a0.dk, a0.dv, a0.dgate};
    SumArgs sum{};
    int sums = 0;
    auto buffer = [&](int t) -> void * {
        const bool f32 = a0.dtype != DIG_BF16 || t == 3;
        if (k == 1 && f32) return result[t];
        float *p = reinterpret_cast<float *>(buffers);
        buffers += plan.buffer;
        sum.src[sums] = p;
        sum.dst[sums] = result[t];
        sum.f32[sums++] = f32;
        return p;
    };
    a.dtype = DIG_BF16_F32OUT;
    if (backward) {
        a.dq = buffer(0);
        a.dk = buffer(1);
        a.dv = buffer(2);
        a.dgate = static_cast<float *>(buffer(3));
    } else {
        a.out = buffer(0);
    }
    a.accumulate = 0;
    uint32_t dirs = 0;
    int held = 0, left = n;
    for (uint32_t d = 0; d < 4; ++d) {
        if (!(mask >> d & 1)) continue;
        dirs |= d << (2 * held++);
        --left;
        if (held < k && left > 0) continue;
        a.g.dir = (int)d;                             // of a single order
        const dig_status st = sweep_orders(a, backward, held, dirs, elems);
        if (st != DIG_OK) return st;
        a.accumulate = 1;
        dirs = 0;
        held = 0;
    }
    if (sums == 0) return DIG_OK;
    const size_t n8 = elems / 8;
    launch_pdl(sum_orders, dim3((unsigned)((n8 + 255) / 256), sums), dim3(256), 0, a.stream, sum, k, elems, n8);
    return cuda_ok(cudaGetLastError());
}

}  // namespace

dig_status sweep_gla_fwd_multi(const GlaArgs &a, unsigned mask) { return sweep_multi(a, false, mask); }
dig_status sweep_gla_bwd_multi(const GlaArgs &a, unsigned mask) { return sweep_multi(a, true, mask); }

dig_status sweep_gla_fwd(const GlaArgs &a) { return sweep_orders(a, false, 1, (uint32_t)a.g.dir, 0); }
dig_status sweep_gla_bwd(const GlaArgs &a) { return sweep_orders(a, true, 1, (uint32_t)a.g.dir, 0); }

}  // namespace dig
