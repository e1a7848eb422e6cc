"""GPU parity of forward sums whose scan orders share launches (few tiles per sequence): all four side by side, three in
two launches, ragged last tiles, shorter chunks."""
import numpy as np
import pytest
import torch

from paper_2405_18428_b200.inputs import Workload, make_inputs
from sweep_plan import launch_bytes, orders_together
from test_gpu_multi import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 72])
@pytest.mark.parametrize("grid,B,H,chunk,dirs", [
    ((16, 16), 4, 6, 64, (0, 1, 2, 3)),
    ((17, 15), 2, 6, 64, (0, 2, 3)),        # 255 tokens; three orders: a launch of two and one that adds to the first buffer
    ((5, 13), 1, 2, 32, (1, 2)),            # 65 tokens: one row in the second tile
    ((23, 40), 8, 6, 64, (0, 1, 2, 3)),
])
def test_orders_in_one_launch(d, grid, B, H, chunk, dirs):
    wl = Workload("orders", B=B, H=H, grid_h=grid[0], grid_w=grid[1], d_k=d, d_v=d, chunk=chunk, dtype="bf16", backward=True,
                  tau=(16.0, 4.0), seed=81)
    print(_check(wl, dirs))


@pytest.mark.parametrize("dirs", [(0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3)])
@pytest.mark.parametrize("d,grid,B,H", [(64, (32, 32), 8, 6), (64, (24, 24), 4, 6), (72, (20, 20), 2, 16), (72, (16, 16), 4, 6)])
def test_last_launch_needs_more_workspace_than_the_one_before(d, grid, B, H, dirs):
    """Three orders as a pair and a single one whose sequences are cut into more segments: right sums, as many launches as
    planned, and nothing written behind the workspace."""
    import oracle
    from paper_2405_18428_b200 import dig
    from parity import TOL_BF16, oracle_threads, rel_err, to_dev
    L = grid[0] * grid[1]
    assert orders_together(B, H, L, d, 64, 3) == 2 and launch_bytes(B, H, L, d, 64, 1) > launch_bytes(B, H, L, d, 64, 2)
    wl = Workload("orders", B=B, H=H, grid_h=grid[0], grid_w=grid[1], d_k=d, d_v=d, chunk=64, dtype="bf16", tau=(16.0, 4.0), seed=83)
    x = make_inputs(wl, conv=False)
    ref = oracle.gla_fwd_multi(x["q"], x["k"], x["v"], oracle.gate(x["g"], x["tau"]), *grid, dirs, threads=oracle_threads())
    q, k_, v, g = (to_dev(x[n], wl) for n in ("q", "k", "v", "g"))
    gate = dig.dig_gate_logsigmoid(g, x["tau"])
    outs = []
    for f32 in (True, False):
        need = dig.dig_gla_multi_workspace_bytes(B, H, *grid, d, d, 64, dig.DIG_BF16_F32OUT if f32 else dig.DIG_BF16, 0)
        ws = torch.full((need + 65536,), 0x5a, dtype=torch.uint8, device="cuda")
        dig.dig_profile_enable(True)
        try:
            out = dig.dig_gla_fwd_multi(q, k_, v, gate, *grid, dirs, 64, f32_out=f32, workspace=ws[:need])
            launches = dig.dig_profile_read()["sweep_fwd"][0]
        finally:
            dig.dig_profile_enable(False)
        assert dig.dig_last_device_status() == dig.DIG_OK
        assert launches == 2
        assert bool((ws[need:] == 0x5a).all())
        outs.append(out)
    assert rel_err(outs[0].cpu().numpy(), ref) <= TOL_BF16
    assert torch.equal(outs[1], outs[0].to(torch.bfloat16))       # the fp32 sums rounded once


@pytest.mark.parametrize("d,grid,B,H", [(64, (16, 16), 4, 6), (72, (17, 15), 2, 6), (64, (12, 16), 8, 16)])
def test_every_mask_with_the_least_workspace(d, grid, B, H):
    """Orders that would share a launch run one by one where the workspace has room for one order alone; less is refused."""
    import oracle
    from paper_2405_18428_b200 import dig
    from parity import TOL_BF16, oracle_threads, rel_err, to_dev
    L = grid[0] * grid[1]
    assert orders_together(B, H, L, d, 64, 4) > 1
    wl = Workload("orders", B=B, H=H, grid_h=grid[0], grid_w=grid[1], d_k=d, d_v=d, chunk=64, dtype="bf16", tau=(16.0, 4.0), seed=84)
    x = make_inputs(wl, conv=False)
    a = oracle.gate(x["g"], x["tau"])
    ref = [oracle.gla_fwd(x["q"], x["k"], x["v"], a, *grid, i, threads=oracle_threads()) for i in range(4)]
    q, k, v, g = (to_dev(x[n], wl) for n in ("q", "k", "v", "g"))
    gate = dig.dig_gate_logsigmoid(g, x["tau"])
    for f32 in (True, False):
        need = launch_bytes(B, H, L, d, 64, 1) + (0 if f32 else -(-B * L * H * d * 4 // 256) * 256)
        assert need < dig.dig_gla_multi_workspace_bytes(B, H, *grid, d, d, 64, dig.DIG_BF16_F32OUT if f32 else dig.DIG_BF16, 0)
        ws = torch.full((need + 65536,), 0x5a, dtype=torch.uint8, device="cuda")
        for mask in range(1, 16):
            dirs = [i for i in range(4) if mask >> i & 1]
            out = dig.dig_gla_fwd_multi(q, k, v, gate, *grid, dirs, 64, f32_out=f32, workspace=ws[:need])
            want = sum(ref[i] for i in dirs)
            rounding = 0 if f32 else 2.0 ** -9 * abs(want).max() / np.sqrt((want ** 2).mean())      # of the largest value to bf16
            assert rel_err(out.float().cpu().numpy(), want) <= TOL_BF16 + rounding, dirs
        assert dig.dig_last_device_status() == dig.DIG_OK
        assert bool((ws[need:] == 0x5a).all())
        with pytest.raises(dig.DigError) as e:
            dig.dig_gla_fwd_multi(q, k, v, gate, *grid, (0, 1), 64, f32_out=f32, workspace=ws[:4096])
        assert e.value.status == dig.DIG_ERR_WORKSPACE
