"""Results stored in 32-byte sectors, and where rows start between them."""
import pytest
import torch

import paper_2001_07710_b200 as pc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("N,H,W,C,F,stride", [(1, 9, 11, 16, 8, 1), (2, 20, 21, 16, 24, 1), (3, 30, 31, 32, 72, 2), (40, 30, 31, 48, 136, 1), (24, 28, 28, 64, 128, 1)])
def test_outputs_at_any_multiple_of_16_bytes(N, H, W, C, F, stride, dtype):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(F)
    tdt, step = (torch.float16, 8) if dtype == "f16" else (torch.float32, 4)
    masks, n_keep = pc.pat_library_builtin(8), F * C // 4
    pid, wm = pc.pat_project(torch.randn((F, C, 3, 3), generator=gen, device="cuda"), masks, n_keep)
    blob = pc.pat_pack(wm, pid, masks, n_keep, dtype)
    x = torch.randn((N, H, W, C), generator=gen, device="cuda").to(tdt)
    shape = (N, (H - 1) // stride + 1, (W - 1) // stride + 1, F)
    n = torch.Size(shape).numel()
    outs = []
    for shift in (0, step):
        buf = torch.full((n + 64,), 7.0, dtype=tdt, device="cuda")
        y = buf[16 + shift:16 + shift + n].view(shape)
        pc.pat_conv3x3(blob, F, C, masks, n_keep, dtype, x, stride, y=y, relu=True)
        assert pc.pat_query_status() == 0
        assert bool((buf[:16 + shift] == 7.0).all()) and bool((buf[16 + shift + n:] == 7.0).all())
        outs.append(y)
    assert torch.equal(outs[0], outs[1])
    # against a float64 convolution: a rounding of the result in fp16; sums off by a step of 2^-23 per term at most
    wd = pc.pat_unpack(blob, F, C, masks, n_keep, dtype).double()
    conv = lambda a, b: torch.nn.functional.conv2d(a.permute(0, 3, 1, 2).double(), b, stride=stride, padding=1).permute(0, 2, 3, 1)
    ref, mag = conv(x, wd).clamp(min=0), conv(x.abs(), wd.abs())
    bound = 4 * C * 2.0 ** -23 * mag + (2.0 ** -11 * ref.abs() + 2.0 ** -25 if dtype == "f16" else 0.0)
    assert bool(((outs[0].double() - ref).abs() <= bound).all())
