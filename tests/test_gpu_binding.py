"""What the compiled binding hands to the library: scratch memory is checked before any kernel is launched on it, sets of
scan orders keep their bits."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _calls(dig):
    B, gh, gw, H, d = 1, 8, 8, 2, 64
    g = torch.Generator(device="cuda").manual_seed(1)
    t = [torch.randn(B, gh * gw, H, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(4)]
    q, k, v, dO = t
    gate = torch.full((B, gh * gw, H, d), -0.05, device="cuda")
    s = torch.zeros(B, H, d, d, device="cuda")
    return {
        "fwd": lambda **w: dig.dig_gla_fwd(q, k, v, gate, gh, gw, **w),
        "bwd": lambda **w: dig.dig_gla_bwd(q, k, v, gate, dO, gh, gw, **w),
        "fwd_state": lambda **w: dig.dig_gla_fwd_state(q, k, v, gate, s, gh, gw, **w),
        "bwd_state": lambda **w: dig.dig_gla_bwd_state(q, k, v, gate, dO, s, s, gh, gw, **w),
        "fwd_multi": lambda **w: dig.dig_gla_fwd_multi(q, k, v, gate, gh, gw, range(4), **w),
        "bwd_multi": lambda **w: dig.dig_gla_bwd_multi(q, k, v, gate, dO, gh, gw, range(4), **w),
        "fwd_beta": lambda **w: dig.dig_gla_fwd_beta(q, k, v, gate, gate, gh, gw, **w),
        "bwd_beta": lambda **w: dig.dig_gla_bwd_beta(q, k, v, gate, gate, dO, gh, gw, **w),
        "fwd_outgate": lambda **w: dig.dig_gla_fwd_outgate(q, k, v, gate, dO, gh, gw, **w),
        "outgate_bwd": lambda **w: dig.dig_gla_outgate_bwd(q, k, dO, **w),
        "conv_bwd": lambda **w: dig.dig_srem_dwconv_bwd(q.view(B, gh * gw, -1), torch.zeros(3, 3, H * d, device="cuda", dtype=q.dtype),
                                                        k.view(B, gh * gw, -1), gh, gw, **w),
    }


@pytest.mark.parametrize("call", ["fwd", "bwd", "fwd_state", "bwd_state", "fwd_multi", "bwd_multi", "fwd_beta", "bwd_beta", "fwd_outgate",
                                  "outgate_bwd", "conv_bwd"])
def test_workspace_has_to_be_dense_device_memory(call):
    from paper_2405_18428_b200 import dig
    f = _calls(dig)[call]
    n = 8 << 20
    with pytest.raises(ValueError, match="workspace: need"):
        f(workspace=torch.empty(n, dtype=torch.uint8))
    with pytest.raises(ValueError, match="workspace: need"):
        f(workspace=torch.empty(2 * n, dtype=torch.uint8, device="cuda")[::2])
    flat = lambda r: [x for x in (r if isinstance(r, tuple) else (r,)) if x is not None]
    for a, b in zip(flat(f()), flat(f(workspace=torch.empty(n, dtype=torch.uint8, device="cuda")))):
        assert torch.equal(a, b)


def test_scan_orders_beyond_the_four_are_the_librarys_refusal():
    from paper_2405_18428_b200 import dig
    q = torch.randn(1, 64, 1, 64, device="cuda").to(torch.bfloat16)
    gate = torch.full(q.shape, -0.05, device="cuda")
    for orders in ([4], [0, 31], []):
        for f in (lambda: dig.dig_gla_fwd_multi(q, q, q, gate, 8, 8, orders), lambda: dig.dig_gla_bwd_multi(q, q, q, gate, q, 8, 8, orders)):
            with pytest.raises(dig.DigError) as e:
                f()
            assert e.value.status == dig.DIG_ERR_INVALID_ARG
