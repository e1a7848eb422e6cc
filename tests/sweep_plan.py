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
BACKWARD = ((14, 54), (32, 23), (88, 95), (62, 73), 67, {32: 133, 16: 280}, 150)


def costed_plan(sequences: int, ntile: int, backward: bool, chunk: int = 64, d: int = 64, limit: int | None = None) -> tuple[int, int, int]:
    """(segments per sequence, tiles per segment, cost); limit: bytes that forward passes in chunks above 64 keep to."""
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
    return -(-ntile // best_g), best_g, best


def sweep_plan(*args, **kw) -> tuple[int, int]:
    """(segments per sequence, tiles per segment)."""
    return costed_plan(*args, **kw)[:2]


def orders_together(B: int, H: int, L: int, d: int, chunk: int, orders: int) -> int:
    """Scan orders that share a launch of a forward sum (chunks of up to 64)."""
    elems, best, k, j = B * L * H * d, None, 1, 1
    launch = lambda n: costed_plan(B * H * n, -(-L // 64), False, chunk, d)[2] if n else 0
    while j <= orders and (j == 1 or elems * j < 1 << 31):
        cost = launch(j) * (orders // j) + launch(orders % j)
        if j > 1:
            cost += 100 * (2 * j - 1) * 4 * elems // 600000 + 2000
        if best is None or cost < best:
            best, k = cost, j
        j *= 2
    return k


def launch_bytes(B: int, H: int, L: int, d: int, chunk: int, orders: int) -> int:
    """Workspace of one launch of so many orders of a forward sum, without the buffers of the results."""
    nseg, _ = sweep_plan(B * H * orders, -(-L // 64), False, chunk, d)
    return segment_bytes(B * H * orders * nseg, d)


def multi_bytes(B: int, H: int, L: int, d: int, chunk: int, orders: int, bf16_out: bool) -> int:
    """Workspace of a forward sum over so many orders: the buffers and the largest of its launches."""
    k = orders_together(B, H, L, d, chunk, orders)
    buffers = -(-B * L * H * d * 4 * k // 256) * 256 if k > 1 or bf16_out else 0
    return buffers + max(launch_bytes(B, H, L, d, chunk, n) for n in (k, orders % k) if n)
