"""The tensor-core convolution kernels at the sizes where their tiling can go wrong: tiles that end inside a row, an image
or a strip, partial channel blocks and filter groups, single tiles whose channels are cut among the CTAs of a cluster,
several rounds per CTA pair, stride 2, pooling; every output element against a float64 convolution of the unpacked
weights (torch), inside a guard band."""
import numpy as np
import pytest
import torch
import torch.nn.functional as Fn

import paper_2001_07710_b200 as pc

pytestmark = pytest.mark.gpu

# fp16: one rounding of the result (2^-11 relative at most) on top of fp32 sums of exact products.  A K-term sum of
# products accumulated with at most one unit in the last place (2^-23) of the running magnitude per step is off by
# at most K 2^-23 sum |w x|; K <= 4 C <= 2048 here.
F16_ROUND = 2.0 ** -11
STEP = 2.0 ** -23


def check(case, dtype, use_workspace=True, masks=None):
    """Returns the number of kernels the call launched."""
    N, H, W, C, F, K, keep, stride, act = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(N * 1000 + H * 7 + W + C + F)
    w = torch.randn((F, C, 3, 3), generator=gen, device="cuda") * (2.0 / (9 * C)) ** 0.5
    tdt = torch.float16 if dtype == "f16" else torch.float32
    x = torch.randn((N, H, W, C), generator=gen, device="cuda").clamp_(min=0).to(tdt)
    if masks is None:
        masks = pc.pat_library_builtin(K)
    n_keep = int(F * C * keep)
    pid, wm = pc.pat_project(w, masks, n_keep)
    blob = pc.pat_pack(wm, pid, masks, n_keep, dtype)
    Ho, Wo = (H - 1) // stride + 1, (W - 1) // stride + 1
    shape = (N, Ho // 2, Wo // 2, F) if act == 2 else (N, Ho, Wo, F)
    n = int(np.prod(shape))
    buf = torch.full((n + 4096,), 7.0, dtype=tdt, device="cuda")
    y = buf[2048:2048 + n].view(shape)
    y.fill_(float("nan"))
    before = pc.pat_launch_count()
    pc.pat_conv3x3(blob, F, C, masks, n_keep, dtype, x, stride, y=y, relu=act == 1, pool=act == 2, use_workspace=use_workspace)
    launches = pc.pat_launch_count() - before
    assert pc.pat_query_status() == 0
    wd = pc.pat_unpack(blob, F, C, masks, n_keep, dtype).double()
    conv = lambda a, b: Fn.conv2d(a.permute(0, 3, 1, 2).double(), b, stride=stride, padding=1)
    ref, mag = conv(x, wd), conv(x.abs(), wd.abs())
    if act:
        ref = ref.clamp(min=0)
    if act == 2:
        ref, mag = Fn.max_pool2d(ref, 2), Fn.max_pool2d(mag, 2)
    ref, mag = ref.permute(0, 2, 3, 1), mag.permute(0, 2, 3, 1)
    assert bool(torch.isfinite(y).all())
    bound = 4 * C * STEP * mag
    if dtype == "f16":
        bound = bound + F16_ROUND * ref.abs() + 2.0 ** -25       # half the smallest subnormal step
    err = (y.double() - ref).abs()
    assert bool((err <= bound).all()), float((err - bound).max())
    assert bool((buf[:2048] == 7.0).all()) and bool((buf[2048 + n:] == 7.0).all())
    return launches


CASES = [
    # N, H, W, C, F, K, keep, stride, act
    (1, 1, 1, 8, 8, 4, 1.0, 1, 0),            # one position, one partial channel block, one partial group
    (1, 14, 14, 64, 64, 8, 0.125, 1, 0),      # less than one tile
    (1, 16, 16, 64, 64, 8, 0.125, 1, 0),      # images end next to a tile's edge (17 rows of 17 positions)
    (5, 7, 7, 512, 512, 8, 0.25, 1, 1),       # channels cut among CTAs
    (1, 14, 14, 512, 512, 8, 0.125, 1, 2),    # the same with pooling
    (2, 60, 61, 64, 64, 8, 0.125, 1, 0),      # the longest rows that are one strip
    (2, 28, 112, 48, 96, 8, 0.25, 1, 2),      # two strips, partial channel block
    (1, 3, 200, 24, 40, 12, 0.25, 1, 0),      # strips longer than the image is high
    (1, 6, 190, 24, 40, 8, 0.25, 2, 0),
    (3, 15, 23, 48, 80, 12, 0.5, 2, 1),       # stride 2, odd sizes
    (3, 14, 14, 256, 256, 8, 0.25, 2, 1),
    (2, 224, 224, 64, 64, 8, 0.125, 1, 2),    # several rounds per pair, weights resident
    (24, 56, 56, 128, 256, 8, 0.125, 1, 0),   # several rounds per pair, two accumulator sets
    (16, 28, 28, 256, 512, 8, 0.125, 1, 1),
    (2, 90, 90, 72, 136, 8, 0.25, 1, 0),      # a second, short channel block; an uneven last group
    (6, 37, 61, 48, 80, 12, 0.25, 1, 1),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(v) for v in c))
def test_f16(case):
    assert check(case, "f16") == 1


@pytest.mark.parametrize("case", CASES + [(8, 28, 28, 256, 256, 4, 1.0, 1, 0), (2, 13, 13, 40, 72, 8, 0.25, 1, 0)], ids=lambda c: "-".join(str(v) for v in c))
def test_f32(case):
    # kept densely enough that the tensor cores run it whatever its size
    assert check(case[:6] + (max(case[6], 0.1875),) + case[7:], "f32") == 1


# fp32 at low density: the workspace kernels' side of the dispatch (stage images, convolution, perhaps a reduction)
@pytest.mark.parametrize("case", [
    (8, 56, 56, 256, 256, 8, 0.1, 1, 0),      # whole items only
    (8, 56, 56, 256, 256, 8, 0.125, 1, 2),
    (8, 14, 14, 512, 512, 8, 0.125, 1, 2),    # every item cut along the channels
    (16, 56, 56, 128, 128, 12, 0.02, 1, 1),   # the ten codes of the twelve patterns
    (8, 56, 56, 1040, 64, 8, 0.03, 1, 0),     # 65 tiles of channels: three words of packed stage bits per filter
], ids=lambda c: "-".join(str(v) for v in c))
def test_f32_low_density(case):
    assert check(case, "f32") >= 2
    assert check(case, "f32", use_workspace=False) == 1 if case[8] == 0 else True


def test_f32_low_density_arbitrary_library():
    masks = np.array([0b000001111, 0b111100000, 0b101000101, 0x03A, 0x0D8, 0b100110001], dtype=np.uint16)
    assert check((24, 56, 56, 256, 128, len(masks), 0.01, 1, 0), "f32", masks=masks) >= 2


def test_entry_point_without_workspace_takes_the_same_kernel():
    assert check((3, 28, 28, 128, 96, 8, 0.125, 1, 0), "f16", use_workspace=False) == 1


@pytest.mark.parametrize("value", [3.4028234e38, -3.4e38, 3.3961e38, 1e-38])
def test_f32_ends_of_the_range(value):
    """Inputs that bf16 would round to infinity, and inputs whose later parts are below the range of bf16."""
    F, C, H = 16, 16, 9
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    w = torch.randn((F, C, 3, 3), generator=gen, device="cuda") * (2.0 ** -8 if abs(value) > 1 else 2.0 ** 20)
    masks = pc.pat_library_builtin(4)
    pid, wm = pc.pat_project(w, masks, F * C)
    blob = pc.pat_pack(wm, pid, masks, F * C, "f32")
    x = torch.zeros((1, H, H, C), device="cuda")
    x[0, 4, 4, 3] = value
    y = pc.pat_conv3x3(blob, F, C, masks, F * C, "f32", x, 1)
    ref = Fn.conv2d(x.permute(0, 3, 1, 2).double(), wm.double(), padding=1).permute(0, 2, 3, 1)
    assert bool(torch.isfinite(y).all())
    # one product per output: the three dropped products of parts are below 2^-25 of it, the sum of the six others is rounded in
    # fp32; parts below 2^-133 (the smallest bf16 step) are lost
    assert bool(((y.double() - ref).abs() <= 6 * STEP * ref.abs() + 2.0 ** -132 * float(w.abs().max())).all())


# near the line between the two fp32 kernels, where estimates with and without pooling would fall on different sides of it
@pytest.mark.parametrize("N,H,C", [(64, 56, 64), (2, 224, 64), (8, 224, 64), (4, 112, 128), (8, 56, 256)])
def test_f32_fused_pooling_has_the_sums_of_the_two_passes(N, H, C):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(N + H + C)
    w = torch.randn((C, C, 3, 3), generator=gen, device="cuda") * (2.0 / (9 * C)) ** 0.5
    x = torch.randn((N, H, H, C), generator=gen, device="cuda").clamp_(min=0)
    masks, n_keep = pc.pat_library_builtin(8), C * C // 8
    pid, wm = pc.pat_project(w, masks, n_keep)
    blob = pc.pat_pack(wm, pid, masks, n_keep, "f32")
    fused = pc.pat_conv3x3(blob, C, C, masks, n_keep, "f32", x, 1, pool=True)
    plain = pc.pat_conv3x3(blob, C, C, masks, n_keep, "f32", x, 1)
    assert torch.equal(fused, pc.pat_relu_maxpool(plain, "f32", True))
    assert torch.equal(pc.pat_conv3x3(blob, C, C, masks, n_keep, "f32", x, 1, relu=True), plain.clamp(min=0))


# unsplit, channels cut among the CTAs of a cluster, several rounds with two accumulator sets, stride 2
NOT_A_NUMBER = [(2, 56, 56, 64, 64, 8, 0.25, 1), (1, 14, 14, 512, 512, 8, 0.25, 1), (16, 28, 28, 64, 256, 8, 0.25, 1), (2, 15, 15, 48, 40, 8, 0.5, 2)]


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("case", NOT_A_NUMBER, ids=lambda c: "-".join(str(v) for v in c))
def test_a_result_that_is_not_a_number_stays_one(case, dtype):
    """Outputs that a kept tap connects to a NaN are NaN without a rectifier; with one (and pooling) they are what
    pat_relu_maxpool makes of that."""
    N, H, W, C, F, K, keep, stride = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(C + F)
    w = torch.randn((F, C, 3, 3), generator=gen, device="cuda") * (2.0 / (9 * C)) ** 0.5
    x = torch.randn((N, H, W, C), generator=gen, device="cuda").clamp_(min=0).to(torch.float16 if dtype == "f16" else torch.float32)
    masks, n_keep = pc.pat_library_builtin(K), int(F * C * keep)
    pid, wm = pc.pat_project(w, masks, n_keep)
    blob = pc.pat_pack(wm, pid, masks, n_keep, dtype)
    x[N - 1, 6, 7, 3] = x[0, 0, 0, C - 1] = float("nan")
    call = lambda **kw: pc.pat_conv3x3(blob, F, C, masks, n_keep, dtype, x, stride, **kw)
    y = call()
    kept = (pc.pat_unpack(blob, F, C, masks, n_keep, dtype) != 0).double()
    touched = Fn.conv2d(torch.isnan(x).permute(0, 3, 1, 2).double(), kept, stride=stride, padding=1).permute(0, 2, 3, 1) > 0
    assert int(touched.sum()) > F // 4
    assert bool(torch.isnan(y[touched]).all())
    assert torch.equal(call(relu=True), pc.pat_relu_maxpool(y, dtype, False))
    if stride == 1:
        assert torch.equal(call(pool=True), pc.pat_relu_maxpool(y, dtype, True))
    assert pc.pat_query_status() == 0


@pytest.mark.parametrize("C,channel", [(32, 5), (32, 20), (64, 40), (72, 70)])
def test_f32_one_product_per_output(C, channel):
    """One non-zero channel in either half of a block of 32 and in a short last one: each output is at most four products, so
    that every one of the six products of parts shows."""
    F, H = 48, 12
    gen = torch.Generator(device="cuda")
    gen.manual_seed(C + channel)
    w = torch.randn((F, C, 3, 3), generator=gen, device="cuda")
    masks = pc.pat_library_builtin(4)
    pid, wm = pc.pat_project(w, masks, F * C)
    blob = pc.pat_pack(wm, pid, masks, F * C, "f32")
    x = torch.zeros((2, H, H, C), device="cuda")
    x[:, ::3, ::3, channel] = torch.randn((2, H // 3, H // 3), generator=gen, device="cuda")       # three apart: one product each
    y = pc.pat_conv3x3(blob, F, C, masks, F * C, "f32", x, 1)
    ref = Fn.conv2d(x.permute(0, 3, 1, 2).double(), wm.double(), padding=1).permute(0, 2, 3, 1)
    # three products of parts left out, below 2^-25 together; six added up with at most a unit in the last place each
    assert bool(((y.double() - ref).abs() <= 6 * STEP * ref.abs()).all())


@pytest.mark.parametrize("value", [3.4028234e38, -3.4e38, 3.3961e38])
def test_f32_largest_weights(value):
    """Weights that bf16 would round to infinity."""
    F, C, H = 16, 16, 9
    gen = torch.Generator(device="cuda")
    gen.manual_seed(6)
    w = torch.randn((F, C, 3, 3), generator=gen, device="cuda")
    w[::2, 5, 1, 1] = value                    # the centre belongs to every built-in mask
    masks = pc.pat_library_builtin(4)
    pid, wm = pc.pat_project(w, masks, F * C)
    blob = pc.pat_pack(wm, pid, masks, F * C, "f32")
    x = torch.zeros((1, H, H, C), device="cuda")
    x[0, 2:7, 2:7, 5] = torch.rand((5, 5), generator=gen, device="cuda") * 2.0 ** -8
    y = pc.pat_conv3x3(blob, F, C, masks, F * C, "f32", x, 1)
    conv = lambda a, b: Fn.conv2d(a.permute(0, 3, 1, 2).double(), b.double(), padding=1).permute(0, 2, 3, 1)
    ref, mag = conv(x, wm), conv(x.abs(), wm.abs())
    assert bool(torch.isfinite(y).all())
    # at most four products per output (one channel, four taps), each with three dropped products of parts below 2^-25 of it
    assert bool(((y.double() - ref).abs() <= 6 * STEP * mag).all())


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("case", NOT_A_NUMBER + [(1, 10, 130, 72, 136, 12, 0.5, 1)], ids=lambda c: "-".join(str(v) for v in c))
def test_an_infinite_input_reaches_only_the_kept_taps(case, dtype):
    """The tensor cores run removed taps as zeros: an infinity or NaN of the input must not come through them."""
    N, H, W, C, F, K, keep, stride = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(C * F)
    w = torch.randn((F, C, 3, 3), generator=gen, device="cuda") * (2.0 / (9 * C)) ** 0.5
    x = torch.randn((N, H, W, C), generator=gen, device="cuda").clamp_(min=0).to(torch.float16 if dtype == "f16" else torch.float32)
    masks, n_keep = pc.pat_library_builtin(K), int(F * C * keep)
    pid, wm = pc.pat_project(w, masks, n_keep)
    blob = pc.pat_pack(wm, pid, masks, n_keep, dtype)
    x[N - 1, 6, 7, 3] = x[0, 0, 0, C - 1] = x[0, H - 1, W - 1, 0] = x[0, 8, 4, 5] = float("inf")
    x[0, 9, 5, 20] = -float("inf")             # with its neighbour of the other sign: some outputs read both
    x[N - 1, 3, W - 1, 9] = float("nan")
    call = lambda **kw: pc.pat_conv3x3(blob, F, C, masks, n_keep, dtype, x, stride, **kw)
    y = call()
    wd = pc.pat_unpack(blob, F, C, masks, n_keep, dtype).double()
    conv = lambda a, b: Fn.conv2d(a.permute(0, 3, 1, 2).double(), b.double(), stride=stride, padding=1).permute(0, 2, 3, 1)
    finite = torch.where(torch.isfinite(x), x, torch.zeros_like(x))
    up = conv(torch.isposinf(x), wd > 0) + conv(torch.isneginf(x), wd < 0) > 0.5
    down = conv(torch.isposinf(x), wd < 0) + conv(torch.isneginf(x), wd > 0) > 0.5
    none = (conv(torch.isnan(x), wd != 0) > 0.5) | (up & down)
    up, down = up & ~none, down & ~none
    assert int(none.sum()) and int(up.sum()) and int(down.sum())
    assert torch.equal(torch.isnan(y), none) and torch.equal(torch.isposinf(y), up) and torch.equal(torch.isneginf(y), down)
    ref, mag = conv(finite, wd), conv(finite.abs(), wd.abs())
    bound = 4 * C * STEP * mag + (F16_ROUND * ref.abs() + 2.0 ** -25 if dtype == "f16" else 0.0)
    assert bool(((y.double() - ref).abs() <= bound)[~(none | up | down)].all())
    assert torch.equal(call(relu=True), pc.pat_relu_maxpool(y, dtype, False))
    if stride == 1 and H % 2 == 0 and W % 2 == 0 and pc.pat_conv3x3_workspace(F, C, dtype, N, H, W, 1):
        assert torch.equal(call(pool=True), pc.pat_relu_maxpool(y, dtype, True))
    assert pc.pat_query_status() == 0
    x.fill_(float("nan"))                      # every output is formed again
    assert torch.equal(torch.isnan(call()), conv(torch.ones_like(x), wd != 0) > 0.5) and pc.pat_query_status() == 0


# CTA pairs over whole sums, one round and several; channels cut among the CTAs of a cluster; a short last chunk
@pytest.mark.parametrize("case", [(64, 28, 28, 4608, 64), (16, 28, 28, 1096, 256), (64, 14, 14, 2560, 320), (1, 14, 14, 8192, 64)], ids=lambda c: "-".join(str(v) for v in c))
def test_f16_long_sums_do_not_drift(case):
    """Positive data: a sum that only ever drops bits ends low by a share that grows with its length."""
    N, H, W, C, F = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(C)
    w = torch.rand((F, C, 3, 3), generator=gen, device="cuda") / C
    x = torch.rand((N, H, W, C), generator=gen, device="cuda").to(torch.float16)
    masks = pc.pat_library_builtin(4)
    pid, wm = pc.pat_project(w, masks, F * C)
    blob = pc.pat_pack(wm, pid, masks, F * C, "f16")
    y = pc.pat_conv3x3(blob, F, C, masks, F * C, "f16", x, 1)
    assert pc.pat_query_status() == 0
    wd = pc.pat_unpack(blob, F, C, masks, F * C, "f16").double()
    low, total, n = 0.0, 0.0, 0
    for i in sorted({0, N // 2, N - 1}):
        ref = Fn.conv2d(x[i:i + 1].permute(0, 3, 1, 2).double(), wd, padding=1).permute(0, 2, 3, 1)
        err = y[i:i + 1].double() - ref
        # 512 channels are 288 steps; a step drops less than two units in the last place of its running sum
        assert bool((err.abs() <= (F16_ROUND + 288 * 2 * STEP) * ref).all())
        low, total, n = low + float(err.sum()), total + float(ref.sum()), n + ref.numel()
    # in the mean one of the two, of a running sum that is half of the whole in the mean; roundings of the results (at most
    # 2^-11, either way) leave five of their standard deviations
    assert abs(low) <= (288 * STEP / 2 + 5 * F16_ROUND / (3 * n) ** 0.5) * total


# every way in which the kernels are run: weights resident, CTA pairs over a ring, channels cut among a cluster's CTAs, sums over
# several chunks; fp32 pairs and clusters; with pooling, whose epilogue warps meet at barriers
@pytest.mark.parametrize("dtype,case", [("f16", (4, 56, 56, 64, 64, 8, 0.125, 1, 0)), ("f16", (24, 28, 28, 256, 512, 8, 0.125, 1, 1)),
                                        ("f16", (1, 14, 14, 512, 512, 8, 0.125, 1, 2)), ("f16", (16, 28, 28, 1096, 256, 8, 0.125, 1, 0)),
                                        ("f32", (24, 28, 28, 256, 256, 8, 0.25, 1, 2)), ("f32", (1, 14, 14, 512, 512, 8, 0.25, 1, 0)),
                                        ("f32", (4, 29, 29, 64, 64, 8, 0.25, 2, 1))], ids=str)
def test_a_wait_that_runs_out_ends_the_kernel(dtype, case):
    """The weights of one stage are never copied (test hook) and the waits are limited to 1 ms: the call ends by itself with a
    status, and the next one is correct."""
    N, H, W, C, F, K, keep, stride, act = case
    masks, n_keep = pc.pat_library_builtin(K), int(F * C * keep)
    pid, wm = pc.pat_project(torch.ones((F, C, 3, 3), device="cuda"), masks, n_keep)
    blob = pc.pat_pack(wm, pid, masks, n_keep, dtype)
    x = torch.ones((N, H, W, C), dtype=torch.float16 if dtype == "f16" else torch.float32, device="cuda")
    try:
        pc.pat_debug_set(0, 1_000_000)
        pc.pat_debug_set(1, 1)
        pc.pat_conv3x3(blob, F, C, masks, n_keep, dtype, x, stride, relu=act == 1, pool=act == 2)
        with pytest.raises(pc.PatError) as e:
            pc.pat_query_status()
        assert e.value.code == 9
    finally:
        pc.pat_debug_set(1, -1)
        pc.pat_debug_set(0, 0)
    assert pc.pat_query_status() == 0
    check(case, dtype)
