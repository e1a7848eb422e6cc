"""The cut of the tcgen05 kernels restated: how many segments of how many 64-token tiles a sequence is worked in (148 SMs,
two CTAs per SM).  Tests that mean to reach a certain cut assert it through this; tests/test_sweep_plan.py holds the
restatement against the library's workspace sizes."""


def sweep_plan(sequences: int, ntile: int, backward: bool) -> tuple[int, int]:
    """(segments per sequence, tiles per segment)"""
    slots, best, best_g = 148 * 2, None, ntile
    nseg, g = 1, ntile
    while True:
        cost = -(-sequences * nseg // slots) * (g + 1) * 10
        if nseg > 1:
            cost += 15 if backward else cost // 2 + 30
        if best is None or cost < best:
            best, best_g = cost, g
        if g == 1:
            break
        nseg = -(-ntile // (g - 1))
        g = -(-ntile // nseg)
    return -(-ntile // best_g), best_g
