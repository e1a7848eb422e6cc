"""GPU parity of the fp32 kernels where several CTAs share a chunk (few chunks): slices of 2 and 4 of the key channels, two
parts of the rows, the edges of the rule and ragged last chunks."""
import pytest

from paper_2405_18428_b200.inputs import Workload
from parity import check_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_k,d_v,chunk,L,H", [
    (64, 64, 64, 1, 1),             # one token
    (64, 64, 64, 256, 6),           # 24 chunks: four slices, two parts
    (64, 64, 64, 64 * 18, 2),       # 36 chunks: two slices, two parts
    (64, 64, 64, 64 * 18 + 1, 2),   # 38 chunks: two slices, one part
    (64, 64, 64, 64 * 49 - 7, 1),   # 49 chunks: two slices in the backward pass alone
    (64, 64, 64, 64 * 37 - 5, 2),   # 74 chunks: none
    (64, 64, 64, 64 * 37 + 3, 2),
    (72, 72, 64, 64 * 37 - 5, 2),   # wide heads: 74 chunks share, 72 channels are cut in two at most
    (72, 72, 64, 64 * 37 + 3, 2),   # 76 do not
    (72, 72, 32, 100, 3),
    (80, 80, 64, 64 * 8 + 9, 1),    # four slices of 20 channels
    (16, 24, 128, 128 * 29 + 40, 2),        # 60 chunks: four slices, two parts
    (16, 32, 16, 40, 2),
    (24, 16, 128, 200, 1),          # scores in a place of their own
])
def test_shared_chunks(d_k, d_v, chunk, L, H):
    wl = Workload("shared", B=1, H=H, grid_h=1, grid_w=L, d_k=d_k, d_v=d_v, chunk=chunk, dtype="f32", backward=True, tau=(16.0, 4.0), seed=82)
    print(check_workload(wl, 1))
