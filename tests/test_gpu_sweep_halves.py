"""GPU parity of the sweep kernels on tiles worked as two 32-row sub-chunks in one pass: last tiles that end around
the middle, tiles of either kind side by side, short and uncut sequences, with a start state and its gradient."""
import pytest

from paper_2405_18428_b200.inputs import Workload
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
