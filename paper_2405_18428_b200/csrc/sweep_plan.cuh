// Host side of the tcgen05 sweep kernels: how a pass is cut into segments, which scan orders share a launch, and what workspace
// that takes.  Plain arithmetic without CUDA calls.
#pragma once

#include "sweep.cuh"

namespace dig {
namespace sw {

constexpr int kPerSm = 2;       // CTAs of 256 threads that share an SM, for every kernel of the family

struct SweepWs {
    float *seg_state, *seg_gamma, *seg_dstate, *seg_carry, *slot_g;
    __half *seg_state16, *slot_s;
    size_t bytes;
};
inline SweepWs carve(char *base, const Geom &g, const Plan &pl, bool backward)
{
    SweepWs w{};
    const size_t segs = (size_t)g.B * g.H * pl.nseg, dd = (size_t)g.dk * g.dv;
    size_t o = 0;
    auto take = [&](size_t bytes) { char *p = base + o; o += align256(bytes); return p; };
    w.seg_state = reinterpret_cast<float *>(take(segs * dd * 4));
    w.seg_gamma = reinterpret_cast<float *>(take(segs * g.dk * 4));
    if (backward) {
        const size_t slots = (size_t)kSlots * g.B * g.H * pl.ntile;
        w.seg_dstate = reinterpret_cast<float *>(take(segs * dd * 4));
        w.seg_carry = reinterpret_cast<float *>(take(segs * g.dk * 4));
        w.seg_state16 = reinterpret_cast<__half *>(take(segs * dd * 2));
        w.slot_s = reinterpret_cast<__half *>(take(slots * dd * 2));
        w.slot_g = reinterpret_cast<float *>(take(slots * g.dk * 4));
    }
    w.bytes = o;
    return w;
}

// Segment length.  Cost of a pass in 0.1 us: launches, a fill per round of CTAs, tiles, and the scan.  An SM with one CTA works a
// tile in two thirds of the time that two sharing it take.  Uncut sequences run the forward sweep alone; cut ones also the local
// sweep and the scan; the backward pass needs the local sweep in either case.  Sub-chunks add to the tiles' cost, so short
// sequences in chunks of 16 are cut where whole tiles would not be (3 tiles of 6 sequences, d = 64: 24.4 us uncut, 18.7 cut; chunks
// of 64: 9.1 uncut).  A cut has to win by 2 us (backward: 1), which its launches cost the host where nothing else keeps the device
// busy (a 256-token image: 19.2 us per block uncut, 22.6 cut, although the device is 0.6 us faster).
// Against 3288 measured cuts of 2 to 768 sequences of 2 to 64 tiles, chunks of 16, 32 and 64, d = 64 and 72, gates of temperature
// 16: the cut chosen is 0.1 to 0.6% off the best on average and at most 21% (300 sequences of 6 tiles, d = 72, backward).  The root
// mean square of the cost's error is 5 to 12%; but forward passes in chunks of 32 are charged 190% for a tile that takes 117%
// since two halves share a pass.  That is as close to the best (0.3%; 0.4% with 117), and with heads whose gates need shorter
// sub-chunks it is the safer side: 80 sequences of 16 tiles, d = 72, tau = 2: 114 us, 171 with 117.  Backward passes have the 133 that
// fits (with 170: 480 sequences of 16 tiles, d = 72, 696 us instead of 545).
struct PassCost {
    int fixed[2], round[2], pair[2], alone[2];      // [cut]; pair: a tile on an SM with two CTAs, alone: with one
    int scan;                                       // per machine full of segments
    int chunk32, chunk16, d72;                      // factors of a tile's cost, per cent
};
constexpr PassCost kForward = {{21, 75}, {5, 8}, {32, 51}, {22, 37}, 35, 190, 310, 140};
constexpr PassCost kBackward = {{14, 54}, {32, 23}, {88, 95}, {62, 73}, 67, 133, 280, 150};
// Chunks above 64 tokens: forward plans stay within the scratch of dig_gla_fwd_static where uncut sequences do (the
// same plan serves dig_gla_fwd, so that both give the same bits).  No other family's workspace is counted there that
// would be larger anyway; with chunks of up to 64 the per-chunk states of the other families always are.
inline Plan make_plan(const Geom &g, int sms, int per_sm, bool backward, long long *least = nullptr)
{
    Plan p;
    p.ntile = (g.L + T - 1) / T;
    p.sub_max = g.C < T ? g.C : T;
    p.gh_inv = g.gh > 1 ? (uint32_t)((1ull << 32) / (unsigned)g.gh) : 0xffffffffu;
    const PassCost &c = backward ? kBackward : kForward;
    const long long slots = (long long)sms * per_sm, bh = (long long)g.B * g.H;
    const long long tile = (p.sub_max == 16 ? c.chunk16 : p.sub_max == 32 ? c.chunk32 : 100) * (g.dk == 72 ? c.d72 : 100) / 100;      // per cent
    long long best = -1;
    p.G = p.ntile;
    // the shortest G of every number of segments that occurs (about 2 sqrt(ntile) of them)
    for (int nseg = 1, G = p.ntile;; nseg = (p.ntile + G - 2) / (G - 1), G = (p.ntile + nseg - 1) / nseg) {
        const long long segs = bh * nseg, rest = segs % slots;
        const long long pairs = segs / slots + (rest > sms), alone = rest > 0 && rest <= sms;          // rounds of either kind
        const int cut = nseg > 1;
        const long long cost = 100 * (c.fixed[cut] + (pairs + alone) * c.round[cut]) + tile * G * (pairs * c.pair[cut] + alone * c.alone[cut]) +
                               (cut ? 100 * c.scan * segs / slots : 0);
        p.nseg = nseg;
        const bool fits = backward || g.C <= T || nseg == 1 || carve(nullptr, g, p, false).bytes <= DIG_GLA_STATIC_SCRATCH_BYTES;
        if (best < 0 || (cost < best && fits)) {
            best = cost;
            p.G = G;
        }
        if (G == 1) break;
    }
    p.nseg = (p.ntile + p.G - 1) / p.G;
    if (least) *least = best;
    return p;
}

// Workspace of one launch of `orders` scan orders, without buffers of results.
inline size_t launch_bytes(const Geom &g, int sms, bool backward, int orders, long long *cost = nullptr)
{
    Geom h = g;
    h.B *= orders;
    return carve(nullptr, h, make_plan(h, sms, kPerSm, backward, cost), backward).bytes;
}

// A sum over scan orders: k of them to a launch.  Its workspace has the buffers of bf16 results and of results of several
// orders in front, and behind them what the largest of its launches needs.  A last launch of fewer orders is planned by itself
// and may be cut where the others are not: three orders of 8 x 32 x 32 tokens, 6 heads of 64, are a pair in 1.6 MB and one order
// in 4.8 MB.
struct SumPlan {
    int k;
    size_t buffer;              // bytes of one tensor's buffers
    int buffers;                // tensors that have them
    size_t launch;
    size_t bytes() const { return buffer * buffers + launch; }
};
// Where a sequence has too few tiles to fill the machine, orders of a forward pass side by side need fewer cuts or none, so no
// local sweep and no scan; the results of a launch's orders then stand in buffers of their own, later launches add to them, and
// one pass sums the buffers.  Costs as in make_plan, plus the buffers, written and read at 0.6 MB per 0.1 us, and the summing launch
// (4 us).  bf16 results need the launch and one buffer in any case, fp32 results do not; both are charged half of it, since
// one is to be the other rounded, and the bits depend on the cuts.  On 790 measured sums of 2 to 192 sequences of 1 to 64 tiles
// the grouping is 0.5% off the best on average and 31% faster than one by one, 31 are slower by more than 2% (worst 20%, fp32
// results of 32 sequences of 9 tiles).  768 tiles in 48 sequences, d = 64, four orders: 127 us one after the other, 82 side by side.
// Backward passes keep one order per launch: pairs took 180 instead of 198 us there, but their four tensors' buffers cost as much
// more in the sum.  Offsets of the results have 31 bits.
class SumPlans {
    const Geom &g;
    const bool backward, narrow;
    size_t elems, launch[3];    // of launches of 1, 2 and 4 orders
    long long cost[3];
    int sizes;

public:
    SumPlans(const Geom &geom, int sms, bool bwd, int dtype) : g(geom), backward(bwd), narrow(dtype == DIG_BF16), elems((size_t)g.B * g.L * g.H * g.dk)
    {
        for (sizes = 0; sizes < (backward ? 1 : 3) && (sizes == 0 || elems << sizes < 1ull << 31); ++sizes) launch[sizes] = launch_bytes(g, sms, backward, 1 << sizes, cost + sizes);
    }
    // n orders, the cheapest way whose workspace is at most `limit`; one order per launch where none is
    SumPlan of(int n, size_t limit) const
    {
        SumPlan best{};
        long long least = -1;
        for (int i = 0; i < sizes && 1 << i <= n; ++i) {
            SumPlan p{1 << i, align256(elems * 4 << i), 0, launch[i]};
            p.buffers = backward ? (narrow ? 3 : 0) : (narrow || i > 0);
            if (n == 3 && i == 1 && launch[0] > launch[1]) p.launch = launch[0];          // the third order's launch
            long long c = cost[i] * (n / p.k) + (n % p.k ? cost[0] : 0);                  // three orders: a pair and one
            if (i > 0) c += (long long)(100 * (2 * p.k - 1) * 4 * elems / 600000) + 2000;
            if (least < 0 || (c < least && p.bytes() <= limit)) {
                least = c;
                best = p;
            }
        }
        return best;
    }
};

}  // namespace sw
}  // namespace dig
