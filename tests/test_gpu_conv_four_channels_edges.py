"""Layers whose channels are an odd multiple of four (kernels of their own: other barriers, warps and copies) where things go wrong:
infinities and NaN, blobs of other layers, waits that run out.  And the generic kernel, which runs what the tensor cores do not."""
import pytest
import torch

import paper_2001_07710_b200 as pc
import test_gpu_conv_mma as mma

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("case", [
    (2, 15, 15, 28, 40, 8, 0.5, 2),
    (3, 12, 8, 36, 24, 8, 0.5, 1),            # few columns
    (1, 10, 130, 76, 136, 12, 0.5, 1),        # strips
    (1, 14, 14, 508, 512, 8, 0.25, 1),        # channels cut among the CTAs of a cluster
    (16, 28, 28, 84, 256, 8, 0.25, 1),        # pairs, several rounds
], ids=lambda c: "-".join(str(v) for v in c))
def test_an_infinite_input_reaches_only_the_kept_taps(case, dtype):
    mma.test_an_infinite_input_reaches_only_the_kept_taps(case, dtype)


@pytest.mark.parametrize("dtype,case", [("f16", (4, 56, 56, 36, 64, 8, 0.125, 1, 0)), ("f16", (24, 28, 28, 260, 512, 8, 0.125, 1, 1)),
                                        ("f16", (1, 14, 14, 508, 512, 8, 0.125, 1, 0)), ("f16", (16, 28, 28, 1100, 256, 8, 0.125, 1, 0)),
                                        ("f32", (24, 28, 28, 260, 256, 8, 0.25, 1, 0)), ("f32", (1, 14, 14, 508, 512, 8, 0.25, 1, 0)),
                                        ("f32", (4, 29, 29, 68, 64, 8, 0.25, 2, 1))], ids=str)
def test_a_wait_that_runs_out_ends_the_kernel(dtype, case):
    mma.test_a_wait_that_runs_out_ends_the_kernel(dtype, case)


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("N,H,C,F", [(1, 9, 20, 40), (1, 14, 508, 512), (24, 28, 84, 256)])
def test_the_blob_of_another_library_is_refused(N, H, C, F, dtype):
    masks, other, n_keep = pc.pat_library_builtin(8), pc.pat_library_builtin(8)[::-1].copy(), F * C // 4
    pid, wm = pc.pat_project(torch.ones((F, C, 3, 3), device="cuda"), masks, n_keep)
    blob = pc.pat_pack(wm, pid, masks, n_keep, dtype)
    x = torch.ones((N, H, H, C), dtype=torch.float16 if dtype == "f16" else torch.float32, device="cuda")
    y = torch.full((N, H, H, F), 7.0, dtype=x.dtype, device="cuda")
    pc.pat_conv3x3(blob, F, C, other, n_keep, dtype, x, 1, y=y)
    with pytest.raises(pc.PatError):
        pc.pat_query_status()
    assert bool((y == 7.0).all())
    pc.pat_conv3x3(blob, F, C, masks, n_keep, dtype, x, 1, y=y)
    assert pc.pat_query_status() == 0 and not bool((y == 7.0).all())


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("case", [
    # filters that are no multiple of eight, channels that are no multiple of four
    (2, 9, 33, 10, 12, 4, 0.5, 1, 0), (3, 17, 20, 16, 20, 8, 0.5, 2, 1), (1, 30, 65, 6, 8, 12, 1.0, 1, 1), (2, 7, 7, 130, 36, 8, 0.25, 2, 0),
    (1, 1, 1, 1, 1, 4, 1.0, 1, 0), (1, 40, 31, 33, 70, 8, 0.1, 1, 0),
], ids=lambda c: "-".join(str(v) for v in c))
def test_generic(case, dtype):
    assert mma.check(case, dtype) == (2 if case[8] else 1)         # the rectifier is a pass of its own
