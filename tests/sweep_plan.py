"""The cut of the tcgen05 kernels restated: how many segments of how many 64-token tiles a sequence is worked in (148 SMs,
two CTAs per SM).  Tests that mean to reach a certain cut assert it through this; tests/test_sweep_plan.py holds the
restatement against the library's workspace sizes."""


def segment_bytes(segments: int, d: int) -> int:
    """Workspace of a forward pass: a state and its decay per segment, blocks of 256 bytes."""
    up = lambda x: -(-x // 256) * 256
    return up(segments * d * d * 4) + up(segments * d * 4)


# per pass: launches, fill per round, a tile beside another CTA, a tile alone (each uncut, cut), scan; per cent for
# chunks of 32 and 16 and for d = 72
FORWARD = ((21, 75), (5, 8), (32, 51), (22, 37), 35, {32: 190, 16: 310}, 140)
BACKWARD = ((14, 54), (32, 23), (88, 95), (62, 73), 67, {32: 170, 16: 280}, 150)


def sweep_plan(sequences: int, ntile: int, backward: bool, chunk: int = 64, d: int = 64, limit: int | None = None) -> tuple[int, int]:
    """(segments per sequence, tiles per segment); limit: bytes that forward passes in chunks above 64 keep to."""
    fixed, fill, pair, alone, scan, sub, d72 = BACKWARD if backward else FORWARD
    tile = sub.get(chunk, 100) * (d72 if d == 72 else 100) // 100
    sms, best, best_g = 148, None, ntile
    nseg, g = 1, ntile
    while True:
        segs, cut = sequences * nseg, int(nseg > 1)
        rounds, rest = divmod(segs, 2 * sms)
        pairs, single = rounds + (rest > sms), int(0 < rest <= sms)
        cost = 100 * (fixed[cut] + (pairs + single) * fill[cut]) + tile * g * (pairs * pair[cut] + single * alone[cut])
        cost += 100 * scan * segs // (2 * sms) if cut else 0
        fits = backward or chunk <= 64 or nseg == 1 or limit is None or segment_bytes(segs, d) <= limit
        if best is None or (cost < best and fits):
            best, best_g = cost, g
        if g == 1:
            break
        nseg = -(-ntile // (g - 1))
        g = -(-ntile // nseg)
    return -(-ntile // best_g), best_g
