"""The cut of the tcgen05 kernels restated: how many segments of how many 64-token tiles a sequence is worked in (148 SMs,
two CTAs per SM).  Tests that mean to reach a certain cut assert it through this; tests/test_sweep_plan.py holds the
restatement against the library's workspace sizes."""


def segment_bytes(segments: int, d: int) -> int:
    """Workspace of a forward pass: a state and its decay per segment, blocks of 256 bytes."""
    up = lambda x: -(-x // 256) * 256
    return up(segments * d * d * 4) + up(segments * d * 4)


def sweep_plan(sequences: int, ntile: int, backward: bool, limit: tuple[int, int] | None = None) -> tuple[int, int]:
    """(segments per sequence, tiles per segment); limit = (bytes, head size) for forward passes in chunks above 64."""
    slots, best, best_g = 148 * 2, None, ntile
    nseg, g = 1, ntile
    while True:
        cost = -(-sequences * nseg // slots) * (g + 1) * 10
        if nseg > 1:
            cost += 15 if backward else cost // 2 + 30
        fits = limit is None or nseg == 1 or segment_bytes(sequences * nseg, limit[1]) <= limit[0]
        if best is None or (cost < best and fits):
            best, best_g = cost, g
        if g == 1:
            break
        nseg = -(-ntile // (g - 1))
        g = -(-ntile // nseg)
    return -(-ntile // best_g), best_g
