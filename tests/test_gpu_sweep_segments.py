"""GPU parity of the sweep kernels where sequences are cut into segments of several tiles: the local sweeps
accumulate over a segment, the last tile of the last segment is ragged, sub-chunks divide its tiles."""
import pytest

from paper_2405_18428_b200.inputs import Workload
from parity import check_workload

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
