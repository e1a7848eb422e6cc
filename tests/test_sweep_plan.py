"""The cut of the tcgen05 kernels as the workspace sizes show it: against its restatement, and against the scratch of
dig_gla_fwd_static, whose limit is what dig_gla_workspace_bytes asks for."""
import pytest

from sweep_plan import segment_bytes, sweep_plan


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
