"""GPU parity of the sweep kernels on tiles worked as two 32-row sub-chunks in one pass: last tiles that end around
the middle, tiles of either kind side by side, short and uncut sequences, with a start state and its gradient."""
import pytest
import torch

from paper_2405_18428_b200 import dig
from paper_2405_18428_b200.inputs import Workload
from sweep_plan import sweep_plan
from test_gpu_state_io import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,direction", [(64, 0), (72, 3)])
@pytest.mark.parametrize("L,B,H,chunk,tau", [
    (32, 1, 2, 32, (16.0,)),             # one sub-chunk: not divided
    (33, 1, 2, 32, (16.0,)),             # one row in the upper half
    (64 * 3 + 33, 2, 3, 32, (16.0, 2.0)),
    (64 * 4 + 31, 2, 3, 32, (4.0,)),     # cut into segments; the last tile is one sub-chunk
    (64 * 9 + 63, 1, 4, 64, (16.0, 3.0, 2.0, 4.0)),      # whole tiles, halves and shorter sub-chunks side by side
    (64 * 4, 40, 8, 64, (4.0, 2.0)),     # uncut forward pass
])
def test_tiles_in_two_halves(d, direction, L, B, H, chunk, tau):
    wl = Workload("halves", B=B, H=H, grid_h=1, grid_w=L, d_k=d, d_v=d, chunk=chunk, dtype="bf16", backward=True, tau=tau, seed=71)
    print(_run(wl, direction, 9))


@pytest.mark.parametrize("d,direction", [(64, 0), (72, 0), (64, 1)])
def test_a_nan_stays_in_its_half(d, direction):
    """Two sub-chunks of a tile meet through the state alone: a NaN in the upper one leaves the rows before it as they were, a
    NaN in the lower one the gradients of the rows behind it."""
    L, H, at = 64 * 5 + 50, 2, 64 * 2
    gen = torch.Generator(device="cuda").manual_seed(91)
    x = {n: torch.randn((1, L, H, d), generator=gen, device="cuda").to(torch.bfloat16) for n in ("q", "k", "v", "dO")}
    gate = dig.dig_gate_logsigmoid(torch.randn((1, L, H, d), generator=gen, device="cuda"), [16.0] * H)
    rows = lambda lo, hi: slice(lo, hi) if direction == 0 else slice(L - hi, L - lo)        # scan positions -> tokens

    def run(**bad):
        y = dict(x)
        for n, p in bad.items():
            y[n] = x[n].clone()
            y[n][:, rows(p, p + 1)] = float("nan")
        out = dig.dig_gla_fwd(y["q"], y["k"], y["v"], gate, 1, L, 32, direction)
        return out, *dig.dig_gla_bwd(y["q"], y["k"], y["v"], gate, y["dO"], 1, L, 32, direction)

    clean, before, behind = run(), rows(0, at + 32), rows(at + 32, L)
    for n in ("k", "v"):
        for got, want, name in zip(run(**{n: at + 40})[:4], clean, ("out", "dq", "dk", "dv")):
            assert torch.equal(got[:, before], want[:, before]), (n, name)
    for n in ("q", "dO"):
        for got, want, name in zip(run(**{n: at + 10}), clean, ("out", "dq", "dk", "dv", "dgate")):
            assert torch.equal(got[:, behind], want[:, behind]), (n, name)


@pytest.mark.parametrize("d,direction", [(64, 0), (72, 1)])
@pytest.mark.parametrize("B,H,tiles", [(1, 6, 5), (10, 10, 3), (25, 8, 4), (10, 10, 5)])
def test_one_pass_gives_the_bits_of_a_pass_per_half(B, H, tiles, d, direction):
    """Gates under which every tile needs two halves, in chunks of 64 (a pass each in the backward sweep and in forward sweeps of up
    to four tiles) and of 32 (one pass), the sequences cut alike."""
    backward_too = sweep_plan(B * H, tiles, True, 64, d) == sweep_plan(B * H, tiles, True, 32, d)
    assert sweep_plan(B * H, tiles, False, 64, d) == sweep_plan(B * H, tiles, False, 32, d) and (backward_too or d == 72)
    L = 64 * tiles - 14
    gen = torch.Generator(device="cuda").manual_seed(92)
    normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda")
    q, k, v, dO = (normal(B, L, H, d).to(torch.bfloat16) for _ in range(4))
    gate = -0.4 - 0.01 * torch.rand((B, L, H, d), generator=gen, device="cuda")      # 32 rows: 18.5 to 18.9 of the limit's 23 (log2), 50 rows: 28.9
    s_in, ds_out = normal(B, H, d, d), normal(B, H, d, d)

    def run(chunk):
        out = dig.dig_gla_fwd_state(q, k, v, gate, s_in, 1, L, chunk, direction)
        return out, dig.dig_gla_bwd_state(q, k, v, gate, dO, s_in, ds_out, 1, L, chunk, direction)

    (f64, b64), (f32, b32) = run(64), run(32)
    assert all(torch.equal(x, y) for x, y in zip(f64, f32))
    if backward_too:
        assert all(torch.equal(x, y) for x, y in zip(b64, b32))
    assert dig.dig_last_device_status() == dig.DIG_OK
