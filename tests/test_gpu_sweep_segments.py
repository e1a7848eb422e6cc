"""GPU parity of the sweep kernels where sequences are cut into segments of several tiles: the local sweeps
accumulate over a segment, the last tile of the last segment is ragged, sub-chunks divide its tiles.  The tests that need
both passes cut assert the cut; in test_segments_of_several_tiles (99 to 108 sequences of 9 or 10 tiles) only the
backward pass is."""
import numpy as np
import pytest
import torch

from paper_2405_18428_b200.inputs import Workload, make_inputs
from parity import check_workload, oracle_threads, rel_err, to_dev
from sweep_plan import sweep_plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,grid,B,H,chunk,tau,direction", [
    (64, (7, 83), 10, 10, 64, (16.0, 1.0), 2),     # 581 tokens, 10 tiles, the last with 5 rows; fast decay divides tiles
    (72, (83, 7), 10, 10, 64, (16.0, 4.0), 3),
    (64, (11, 47), 9, 12, 16, (16.0,), 1),         # every tile in sub-chunks of 16
    (72, (5, 103), 9, 12, 32, (4.0,), 2),          # 515 tokens: three rows in the last tile, a sub-chunk of its own
    (72, (1, 577), 11, 9, 64, (2.0,), 0),          # one row in the last tile
])
def test_segments_of_several_tiles(d, grid, B, H, chunk, tau, direction):
    wl = Workload("seg", B=B, H=H, grid_h=grid[0], grid_w=grid[1], d_k=d, d_v=d, chunk=chunk, dtype="bf16", backward=True,
                  tau=tau, seed=61)
    print(check_workload(wl, direction))


@pytest.mark.parametrize("d,tiles,last", [(64, 8, 64), (64, 9, 1), (64, 33, 60), (72, 9, 64), (72, 19, 33), (72, 37, 64)])
def test_scans_over_few_and_many_segments(d, tiles, last):
    """One tile per segment: the scan over segment ends at the edges of its two kernels and of their passes."""
    wl = Workload("scan", B=1, H=2, grid_h=1, grid_w=64 * (tiles - 1) + last, d_k=d, d_v=d, chunk=64, dtype="bf16", backward=True,
                  tau=(16.0, 4.0), seed=62)
    print(check_workload(wl, 1))


@pytest.mark.parametrize("d", [64, 72])
@pytest.mark.parametrize("case", ["small", "far"])
def test_states_of_segments_keep_their_relative_precision(d, case):
    """What a segment of six tiles hands on is accurate relative to its own size, whatever that is: with keys and queries of
    size 1e-5, and with keys only in the first tile of the last segment (and queries only in the last tile of the first one),
    whose products decay by 2^-23 before the segment's end (start).  Bound: operands in fp16, centred per tile, so the
    quantum 2^-25 stays 2^-4 or better of a key of 1e-5 = 2^-16.6 at the tile's weak end (gates of a tile sum to 2^4.7, so
    2^-21) and 2^-12 at its strong end; over the 64 x 6 tokens of a sum, weighted with their decay, that is below 1e-2 of the
    result's RMS (emulated: 3.5e-3; one operand exponent for the whole segment: 2.5e-2, and 0.8 where keys are far)."""
    import oracle
    from paper_2405_18428_b200 import dig
    wl = Workload("prec", B=4, H=12, grid_h=25, grid_w=91, d_k=d, d_v=d, chunk=64, dtype="bf16", backward=True, tau=(16.0,), seed=63)
    assert sweep_plan(48, 36, False, 64, d) == sweep_plan(48, 36, True, 64, d) == (6, 6) and -(-wl.L // 64) == 36
    x = make_inputs(wl, conv=False)
    if case == "small":
        for n in ("q", "k"):
            x[n] = torch.from_numpy(x[n] * np.float32(1e-5)).to(torch.bfloat16).float().numpy()
    else:
        x["k"][:, :30 * 64] = 0.0
        x["k"][:, 31 * 64:] = 0.0
        x["q"][:, :5 * 64] = 0.0
        x["q"][:, 6 * 64:] = 0.0
    q, k, v, g, dO = (to_dev(x[n], wl) for n in ("q", "k", "v", "g", "dO"))
    gate = dig.dig_gate_logsigmoid(g, x["tau"])
    a = gate.double().cpu().numpy()
    thr = oracle_threads()
    _, s_ref = oracle.gla_fwd_state(x["q"], x["k"], x["v"], a, None, wl.grid_h, wl.grid_w, 0, threads=thr)
    ds_ref = oracle.gla_bwd_state(x["q"], x["k"], x["v"], a, x["dO"], None, None, wl.grid_h, wl.grid_w, 0, threads=thr)[4]
    _, s_out = dig.dig_gla_fwd_state(q, k, v, gate, None, wl.grid_h, wl.grid_w, 64, 0)
    ds_in = dig.dig_gla_bwd_state(q, k, v, gate, dO, None, None, wl.grid_h, wl.grid_w, 64, 0)[4]
    errs = rel_err(s_out.cpu().numpy(), s_ref), rel_err(ds_in.cpu().numpy(), ds_ref)
    print(errs)
    assert max(errs) <= 1e-2, errs


@pytest.mark.parametrize("d,grid,B,H,chunk,tau,direction", [
    (64, (25, 91), 4, 12, 64, (16.0, 1.0), 2),     # 36 tiles in segments of 6, the last with 35 rows; fast decay divides tiles
    (72, (91, 25), 3, 16, 64, (16.0, 2.0), 3),
    (64, (1, 1009), 6, 8, 16, (16.0,), 1),         # 16 tiles in segments of 3, sub-chunks of 16, the last tile with 49 rows
    (72, (17, 57), 4, 12, 32, (1.0,), 2),          # 9 rows in the last tile
    (72, (7, 279), 12, 4, 64, (2.0,), 0),          # 31 tiles: the last segment is one tile of 33 rows
])
def test_both_passes_cut_into_segments_of_several_tiles(d, grid, B, H, chunk, tau, direction):
    """(The gate gradient is a sum over all later tokens of products of 11-bit operands, so its error grows with the length:
    2.1e-2 of RMS for tau = 1 over 1953 tokens; hence tau = 2 on the longest.)"""
    for backward in (False, True):
        nseg, g = sweep_plan(B * H, -(-grid[0] * grid[1] // 64), backward, chunk, d)
        assert nseg > 1 and g > 1
    wl = Workload("cut", B=B, H=H, grid_h=grid[0], grid_w=grid[1], d_k=d, d_v=d, chunk=chunk, dtype="bf16", backward=True,
                  tau=tau, seed=64)
    print(check_workload(wl, direction))


@pytest.mark.parametrize("d,chunk", [(64, 16), (72, 32)])
def test_short_chunks_keep_large_operands_in_range_in_every_kernel(d, chunk):
    """Keys of size 30 times half of a 64-token tile's decay (up to 2^11.5) would saturate in fp16; chunks of 16 or 32 tokens,
    which the caller asked for, keep them in range in the local sweeps too."""
    wl = Workload("large", B=2, H=2, grid_h=41, grid_w=32, d_k=d, d_v=d, chunk=chunk, dtype="bf16", backward=True, tau=(4.0,), seed=65)
    assert sweep_plan(4, 21, False, chunk, d)[0] > 1
    x = make_inputs(wl, conv=False)
    x["k"] = torch.from_numpy(x["k"] * np.float32(30)).to(torch.bfloat16).float().numpy()
    print(check_workload(wl, 3, x=x))


@pytest.mark.parametrize("d", [64, 72])
@pytest.mark.parametrize("chunk,tiles,cut", [(16, 3, True), (16, 5, True), (64, 2, False), (32, 5, True)])
def test_short_sequences_are_cut_where_their_chunks_make_them_long(d, chunk, tiles, cut):
    """The forward launches of 6 sequences: a sub-chunk costs most of a tile, the launches of a cut pass stay the same."""
    from paper_2405_18428_b200 import dig
    assert (sweep_plan(6, tiles, False, chunk, d)[0] > 1) == cut
    q = torch.randn(1, 64 * tiles, 6, d, device="cuda").to(torch.bfloat16)
    gate = torch.full(q.shape, -0.05, device="cuda")
    dig.dig_profile_enable(True)
    try:
        dig.dig_gla_fwd(q, q, q, gate, 64, tiles, chunk, 0)
        assert ("sweep_local" in dig.dig_profile_read()) == cut
    finally:
        dig.dig_profile_enable(False)
