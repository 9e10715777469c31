"""fp16 layers whose channels are an odd multiple of four, on images of few columns: the loading warps' lanes take positions of any
row there, rows elsewhere."""
import pytest
import torch

import paper_2001_07710_b200 as pc
from test_gpu_conv_mma import check
from timing import graph_ms

pytestmark = pytest.mark.gpu


# a row has W + 1 positions; one channel step to four in a stage put the line at 20, 10 and 5 of them
@pytest.mark.parametrize("case", [
    (1, 1, 1, 4, 8, 4, 1.0, 2, 0),
    (300, 1, 1, 20, 64, 8, 0.5, 1, 1),        # one-row images, several tiles
    (40, 3, 1, 68, 40, 8, 0.5, 2, 0),         # a second block of one channel step
    (9, 7, 19, 12, 24, 8, 0.5, 1, 0), (9, 7, 20, 12, 24, 8, 0.5, 1, 0),
    (9, 7, 9, 28, 24, 8, 0.5, 1, 1), (9, 7, 10, 28, 24, 8, 0.5, 1, 1),
    (9, 7, 4, 52, 24, 8, 0.5, 1, 0), (9, 7, 5, 52, 24, 8, 0.5, 1, 0),
    (9, 6, 7, 60, 24, 8, 0.5, 2, 0), (9, 6, 9, 60, 24, 8, 0.5, 2, 0),
    (5, 4, 4, 132, 512, 8, 0.25, 1, 0),       # channels cut among the CTAs of a cluster
    (2000, 5, 4, 36, 256, 8, 0.25, 1, 1),     # pairs, several rounds
    (700, 7, 7, 524, 136, 8, 0.2, 2, 0),      # sums of several chunks
], ids=lambda c: "-".join(str(v) for v in c))
def test_f16(case):
    assert check(case, "f16") == 1


@pytest.mark.parametrize("N,H,W,C,F,stride", [(40, 1, 1, 4, 64, 2), (64, 3, 3, 4, 64, 2), (40, 1, 1, 4, 64, 1), (1, 64, 2, 4, 64, 1)])
def test_narrow_images_take_no_longer_than_in_the_general_kernel(N, H, W, C, F, stride):
    """Two channels more take that one.  Its 13 us (stride 2) were 51 with a warp on a row, 9.5 as it is."""
    def ms(C):
        masks, n_keep = pc.pat_library_builtin(4), F * C // 4
        pid, wm = pc.pat_project(torch.ones((F, C, 3, 3), device="cuda"), masks, n_keep)
        blob = pc.pat_pack(wm, pid, masks, n_keep, "f16")
        x = torch.ones((N, H, W, C), dtype=torch.float16, device="cuda")
        y = pc.pat_conv3x3(blob, F, C, masks, n_keep, "f16", x, stride)
        return graph_ms(lambda: pc.pat_conv3x3(blob, F, C, masks, n_keep, "f16", x, stride, y=y))
    ms(C)
    assert ms(C) <= 1.25 * ms(C + 2)
