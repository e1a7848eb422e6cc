"""GPU parity of forward sums whose scan orders share launches (few tiles per sequence): all four side by side, three in
two launches, ragged last tiles, shorter chunks."""
import pytest

from paper_2405_18428_b200.inputs import Workload
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
