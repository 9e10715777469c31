"""Blobs of layers whose channels are an odd multiple of four, packed when such layers had no dense form (their header says how long
they are): the tensor-core kernels find that out and run the generic kernel's tiles."""
import pytest
import torch

import paper_2001_07710_b200 as pc
from timing import graph_ms

pytestmark = pytest.mark.gpu

F16_ROUND, STEP = 2.0 ** -11, 2.0 ** -23


def layer(N, H, W, C, F, K, keep, stride, dtype, old):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(C + F + H)
    masks = pc.pat_library_builtin(K) if K <= 12 else [sum(1 << b for b in c) for c in torch.combinations(torch.arange(9), 4).tolist()][:K]
    n_keep = int(F * C * keep)
    pid, wm = pc.pat_project(torch.randn((F, C, 3, 3), generator=gen, device="cuda") * (2.0 / (9 * C)) ** 0.5, masks, n_keep)
    blob = pc.pat_pack(wm, pid, masks, n_keep, dtype)
    wd = pc.pat_unpack(blob, F, C, masks, n_keep, dtype)
    if old:
        dense = (9 * 2 * (1 if dtype == "f16" else 3) * F * ((C + 7) // 8 * 8) + 255) // 256 * 256
        blob = blob[:blob.numel() - dense].clone()
        blob[32:40].view(torch.int64)[0] = blob.numel()
    x = torch.randn((N, H, W, C), generator=gen, device="cuda").to(torch.float16 if dtype == "f16" else torch.float32)
    return (lambda **kw: pc.pat_conv3x3(blob, F, C, masks, n_keep, dtype, x, stride, **kw)), x, wd


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("case", [
    # N, H, W, C, F, K, keep, stride, relu
    (1, 1, 1, 4, 8, 4, 1.0, 1, False),        # one position; many teams of few warps
    (3, 9, 33, 20, 16, 12, 0.5, 1, True),     # a tile and one more of each axis
    (2, 8, 32, 12, 40, 126, 1.0, 2, True),    # a large library
    (2, 17, 66, 36, 256, 8, 0.25, 2, False),
    (1, 15, 31, 508, 72, 8, 0.02, 1, False),  # channels cut among the CTAs of a cluster; stages without kernels
    (30, 40, 41, 84, 200, 8, 0.2, 1, True),   # pairs, several rounds; filters left over
    (2, 20, 21, 44, 24, 8, 0.0, 1, False),    # nothing kept
    (4, 14, 14, 1036, 96, 8, 0.1, 1, False),
], ids=lambda c: "-".join(str(v) for v in c))
def test_results(case, dtype):
    N, H, W, C, F, K, keep, stride, relu = case
    call, x, wd = layer(*case[:8], dtype, True)
    Ho, Wo = (H - 1) // stride + 1, (W - 1) // stride + 1
    n = N * Ho * Wo * F
    buf = torch.full((n + 4096,), 7.0, dtype=x.dtype, device="cuda")
    y = buf[2048:2048 + n].view(N, Ho, Wo, F)
    y.fill_(float("nan"))
    call(y=y, relu=relu)
    assert pc.pat_query_status() == 0
    conv = lambda a, b: torch.nn.functional.conv2d(a.permute(0, 3, 1, 2).double(), b.double(), stride=stride, padding=1).permute(0, 2, 3, 1)
    ref, mag = conv(x, wd), conv(x.abs(), wd.abs())
    if relu:
        ref = ref.clamp(min=0)
    # one rounding of the result in fp16; 4 C fp32 multiply-adds at most, half a unit of the running magnitude each
    bound = 2 * C * STEP * mag + (F16_ROUND * ref.abs() + 2.0 ** -25 if dtype == "f16" else 0.0)
    assert bool(((y.double() - ref).abs() <= bound).all())
    assert bool((buf[:2048] == 7.0).all()) and bool((buf[2048 + n:] == 7.0).all())
    assert bool(torch.isfinite(layer(*case[:8], dtype, False)[0](relu=relu)).all()) and pc.pat_query_status() == 0      # tensor memory was given back


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("C,F", [(36, 40), (4, 8)])
def test_a_buffer_of_the_former_size_is_packed_without_the_dense_form(C, F, dtype):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(C)
    masks, n_keep = pc.pat_library_builtin(8), F * C // 2
    pid, wm = pc.pat_project(torch.randn((F, C, 3, 3), generator=gen, device="cuda"), masks, n_keep)
    full = pc.pat_pack(wm, pid, masks, n_keep, dtype)
    size = full.numel() - (9 * 2 * (1 if dtype == "f16" else 3) * F * ((C + 7) // 8 * 8) + 255) // 256 * 256
    buf = torch.full((size + 512,), 7, dtype=torch.uint8, device="cuda")
    small = pc.pat_pack(wm, pid, masks, n_keep, dtype, blob=buf[:size])
    assert bool((buf[size:] == 7).all()) and int(small[32:40].view(torch.int64)) == size
    assert torch.equal(pc.pat_unpack(small, F, C, masks, n_keep, dtype), pc.pat_unpack(full, F, C, masks, n_keep, dtype))
    x = torch.randn((2, 9, 10, C), generator=gen, device="cuda").to(torch.float16 if dtype == "f16" else torch.float32)
    y, old = (pc.pat_conv3x3(b, F, C, masks, n_keep, dtype, x, 1) for b in (full, small))
    assert pc.pat_query_status() == 0
    # two sums of up to 2 C terms, rounded to fp16 each
    mag = torch.nn.functional.conv2d(x.abs().permute(0, 3, 1, 2).double(), wm.abs().double(), padding=1).permute(0, 2, 3, 1)
    assert bool(((y.double() - old.double()).abs() <= 4 * C * STEP * mag + (2 * F16_ROUND * y.double().abs() + 2.0 ** -24 if dtype == "f16" else 0.0)).all())
    with pytest.raises(pc.PatError):
        pc.pat_pack(wm, pid, masks, n_keep, dtype, blob=buf[:size - 256])


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("N,H,C,F,stride", [(1, 56, 68, 64, 1), (8, 28, 260, 256, 1), (2, 80, 20, 24, 2)])
def test_time_is_that_of_the_generic_kernel(N, H, C, F, stride, dtype):
    """Two channels more take that kernel.  Measured 0.5 - 1.4 of its time; 10 - 57 times it when every result gathered its own taps."""
    def ms(C, old):
        call, x, _ = layer(N, H, H, C, F, 8, 0.25, stride, dtype, old)
        y = call()
        return graph_ms(lambda: call(y=y), calls=5)
    ms(C + 2, False)
    assert ms(C, True) <= 2.0 * ms(C + 2, False)
    assert pc.pat_query_status() == 0
