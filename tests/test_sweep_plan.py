"""The cut of the tcgen05 kernels as the workspace sizes show it: against its restatement, and against the scratch of
dig_gla_fwd_static, whose limit is what dig_gla_workspace_bytes asks for."""
import os
import subprocess

import pytest

from sweep_plan import multi_bytes, segment_bytes, sweep_plan


@pytest.fixture(scope="module")
def dig():
    from paper_2405_18428_b200 import build, dig
    build.build()
    return dig


SHAPES = [(bh, t) for bh in (1, 6, 16, 43, 48, 64, 80, 100, 160, 300, 700) for t in (1, 2, 5, 16, 31, 36, 64, 72, 101, 196, 256, 400)]


@pytest.mark.parametrize("backward", [False, True])
def test_restated_plan_gives_the_librarys_workspace(dig, backward):
    """d = 72 in chunks of 128, which no other family serves: the sweep workspace alone counts."""
    d, up = 72, lambda x: -(-x // 256) * 256
    for bh, t in SHAPES:
        nseg, _ = sweep_plan(bh, t, backward, 128, d, dig.DIG_GLA_STATIC_SCRATCH_BYTES)
        segs, want = bh * nseg, segment_bytes(bh * nseg, d)
        if backward:
            want += up(segs * d * d * 4) + up(segs * d * 4) + up(segs * d * d * 2) + up(8 * bh * t * d * d * 2) + up(8 * bh * t * d * 4)
        assert dig.dig_gla_workspace_bytes(1, bh, 8, 8 * t, d, d, 128, dig.DIG_BF16, backward) == want, (bh, t)


def test_cutting_sequences_does_not_exceed_the_static_scratch(dig):
    """What fits the 16 MiB array with one state per sequence stays within it however the sequences are cut."""
    limit = dig.DIG_GLA_STATIC_SCRATCH_BYTES
    need = lambda B, H, gh, gw, d: dig.dig_gla_workspace_bytes(B, H, gh, gw, d, d, 128, dig.DIG_BF16, 0)
    assert need(5, 16, 64, 64, 72) <= limit and need(10, 16, 64, 72, 72) <= limit
    for bh, t in SHAPES:
        if segment_bytes(bh, 72) <= limit:
            assert need(1, bh, 8, 8 * t, 72) <= limit, (bh, t)


def test_restated_orders_give_the_librarys_workspace(dig):
    for B, H in [(1, 6), (2, 6), (4, 6), (8, 6), (2, 16), (16, 12)]:
        for t in (1, 2, 3, 5, 7, 9, 16, 20, 36):
            for d in (64, 72):
                for chunk in (16, 32, 64):
                    for dtype in (dig.DIG_BF16, dig.DIG_BF16_F32OUT):
                        want = max(multi_bytes(B, H, 64 * t, d, chunk, n, dtype == dig.DIG_BF16) for n in (1, 2, 3, 4))
                        assert dig.dig_gla_multi_workspace_bytes(B, H, 8, 8 * t, d, d, chunk, dtype, 0) == want, (B, H, t, d, chunk)


def test_launches_of_a_sum_stay_clear_of_its_buffers(tmp_path):
    """The layout itself, compiled from the plan's header: behind the buffers there is room for every launch of a sum, a last
    one of fewer orders among them, which may be cut into more segments than the launches in front of it.  A workspace for one
    order per launch is enough for every sum."""
    from paper_2405_18428_b200 import build
    src = tmp_path / "layout.cu"
    src.write_text(r"""
#include <cstdio>
#include "sweep_plan.cuh"
using namespace dig;
using namespace dig::sw;
int main()
{
    long short_last = 0, over = 0, fewer = 0;
    for (int B : {1, 2, 4, 8, 16, 40}) for (int H : {1, 6, 12, 16}) for (int t = 1; t <= 64; ++t)
    for (int d : {64, 72}) for (int C : {16, 32, 64, 128}) for (int bwd = 0; bwd < 2; ++bwd) for (int dt : {DIG_BF16, DIG_BF16_F32OUT}) {
        Geom g{};
        g.B = B; g.H = H; g.gh = 8; g.gw = 8 * t; g.L = 64 * t; g.dk = g.dv = d; g.C = C; g.N = (g.L + C - 1) / C;
        const SumPlans plans(g, 148, bwd, dt);
        auto bytes = [&](int orders) {
            Geom h = g;
            h.B *= orders;
            return carve(nullptr, h, make_plan(h, 148, kPerSm, bwd), bwd).bytes;
        };
        const size_t one = bytes(1) + (dt == DIG_BF16 ? (bwd ? 3 : 1) * align256((size_t)B * g.L * H * d * 4) : 0);      // one order per launch
        for (int n = 1; n <= 4; ++n) for (size_t limit : {SIZE_MAX, one}) {
            const SumPlan p = plans.of(n, limit);
            over += p.bytes() > limit;
            fewer += limit == one && p.k < plans.of(n, SIZE_MAX).k;
            for (int left = n; left > 0; left -= p.k) {
                const size_t need = bytes(left < p.k ? left : p.k);
                over += p.buffer * p.buffers + need > p.bytes();
                short_last += left < p.k && need > bytes(p.k);
            }
        }
    }
    printf("%ld %ld %ld\n", short_last, over, fewer);
    return 0;
}
""")
    exe = tmp_path / "layout"
    subprocess.run([os.environ.get("NVCC", "nvcc"), *build.NVCC_FLAGS, str(src), "-o", str(exe)], check=True, capture_output=True)
    short_last, over, fewer = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert over == 0
    assert short_last > 100 and fewer > 1000       # sizes at which the last launch needs the most, or orders part, are among them
