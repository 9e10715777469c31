"""Layers whose channels are an odd multiple of four: activation rows that TMA does not take."""
import pytest
import torch

import paper_2001_07710_b200 as pc
from test_gpu_conv_mma import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("case", [
    # N, H, W, C, F, K, keep, stride, act
    (1, 1, 1, 4, 8, 4, 1.0, 1, 0),            # one position, four channels
    (2, 9, 10, 212, 152, 4, 1.0, 1, 1),       # channels cut among the CTAs of a cluster
    (1, 15, 7, 20, 40, 4, 0.5, 1, 0),
    (3, 5, 130, 36, 40, 8, 0.5, 1, 1),        # strips, tiles that start and end inside a row
    (2, 23, 15, 68, 24, 12, 0.3, 2, 0),       # stride 2, a second channel block of four
    (2, 61, 64, 132, 32, 8, 0.25, 2, 1),
    (12, 60, 61, 84, 256, 8, 0.2, 1, 0),      # several rounds, pairs
    (20, 30, 31, 76, 64, 8, 0.2, 1, 1),       # weights resident in fp16
    (4, 14, 14, 1036, 96, 8, 0.2, 1, 0),      # sums of several chunks in fp16
    (90, 30, 30, 524, 136, 8, 0.2, 1, 0),     # the same in pairs
], ids=lambda c: "-".join(str(v) for v in c))
def test_conv(case, dtype):
    assert check(case, dtype) == 1


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("N,H,W,C,F,stride,relu", [(2, 9, 10, 212, 152, 1, True), (1, 7, 7, 20, 40, 1, False), (40, 20, 21, 36, 48, 2, False), (24, 40, 41, 84, 128, 1, True)])
def test_blob_without_dense_form(N, H, W, C, F, stride, relu, dtype):
    """Blobs of these layers once held no dense form; a header says how long its blob is."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(C)
    masks, n_keep = pc.pat_library_builtin(8), F * C // 5
    w = torch.randn((F, C, 3, 3), generator=gen, device="cuda") * (2.0 / (9 * C)) ** 0.5
    pid, wm = pc.pat_project(w, masks, n_keep)
    blob = pc.pat_pack(wm, pid, masks, n_keep, dtype)
    x = torch.randn((N, H, W, C), generator=gen, device="cuda").to(torch.float16 if dtype == "f16" else torch.float32)
    y = pc.pat_conv3x3(blob, F, C, masks, n_keep, dtype, x, stride, relu=relu)
    terms = 1 if dtype == "f16" else 3
    dense = (9 * 2 * terms * F * ((C + 7) // 8 * 8) + 255) // 256 * 256
    old = blob[:blob.numel() - dense].clone()
    old[32:40].view(torch.int64)[0] = old.numel()
    got = pc.pat_conv3x3(old, F, C, masks, n_keep, dtype, x, stride, relu=relu)
    assert pc.pat_query_status() == 0
    # one rounding of the result (fp16), and sums in another order: at most 4 C steps of 2^-23 of the magnitudes added up
    wd = pc.pat_unpack(blob, F, C, masks, n_keep, dtype).double()
    mag = torch.nn.functional.conv2d(x.abs().permute(0, 3, 1, 2).double(), wd.abs(), stride=stride, padding=1).permute(0, 2, 3, 1)
    bound = 8 * C * 2.0 ** -23 * mag + (2.0 ** -10 * y.double().abs() + 2.0 ** -24 if dtype == "f16" else 0.0)
    assert bool(((got.double() - y.double()).abs() <= bound).all())
