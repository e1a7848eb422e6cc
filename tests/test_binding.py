"""The compiled binding rejects what the documented functions do not take, before any kernel is launched."""
import pytest
import torch


@pytest.fixture(scope="module")
def dig():
    from paper_2405_18428_b200 import build, dig
    build.build()
    return dig


def test_cpu_tensors_and_wrong_types_are_rejected(dig):
    t = torch.zeros(1, 4, 1, 64)
    with pytest.raises(ValueError, match="q: need a contiguous CUDA tensor"):
        dig.dig_gla_fwd(t, t, t, t, 2, 2)
    with pytest.raises(ValueError, match="q: need 4 dimensions"):
        dig.dig_gla_bwd(t[0], t, t, t, t, 2, 2)
    with pytest.raises(TypeError, match="unsupported storage type"):
        dig.dig_gla_outgate_fwd(t.double(), t)
    with pytest.raises(TypeError, match="x: need a torch tensor"):
        dig.dig_srem_dwconv(1, t, None, 2, 2)
    with pytest.raises(ValueError, match="x: L != grid_h"):
        dig.dig_srem_dwconv(torch.zeros(1, 4, 8), t, None, 3, 3)
    with pytest.raises(IndexError):
        dig.dig_gate_logsigmoid(t, [16.0, 16.0], t)


def test_cpu_tensors_are_value_errors_where_the_result_is_not_given(dig):
    """The check comes before the result is allocated on the input's device."""
    with pytest.raises(ValueError, match="g: need a contiguous CUDA tensor"):
        dig.dig_gate_logsigmoid(torch.zeros(1, 4, 1, 64), [16.0])
    with pytest.raises(ValueError, match="x: need a contiguous CUDA tensor"):
        dig.dig_srem_dwconv(torch.zeros(1, 4, 8), torch.zeros(3, 3, 8), None, 2, 2)
