"""Packing at the largest channel counts whose lists fit the packing kernel's shared memory, and one beyond."""
import pytest
import torch

import paper_2001_07710_b200 as pc

pytestmark = pytest.mark.gpu


# lists of C bytes and C / 16 words (and C / 16 x K words up to 24 KB) fit 48 KB
@pytest.mark.parametrize("F,C,K,keep,dtype", [(3, 39316, 8, 0.5, "f16"), (32, 39312, 8, 0.1, "f32"), (8, 39312, 4, 1.0, "f32"),
                                              (5, 28080, 2, 0.5, "f16"), (5, 28080, 2, 0.5, "f32"), (3, 38496, 8, 0.25, "f16")])
def test_largest_channel_counts(F, C, K, keep, dtype):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(C + F)
    w = torch.randn((F, C, 3, 3), generator=gen, device="cuda")
    masks, n_keep = [0x03A, 0x0B8] if K == 2 else pc.pat_library_builtin(K), int(F * C * keep)
    pid, wm = pc.pat_project(w, masks, n_keep)
    blob = pc.pat_pack(wm, pid, masks, n_keep, dtype)
    want = wm.half().float() if dtype == "f16" else wm
    assert torch.equal(pc.pat_unpack(blob, F, C, masks, n_keep, dtype), want)
    assert pc.pat_query_status() == 0


def test_one_more_is_refused():
    F, C, masks = 2, 39317, pc.pat_library_builtin(8)
    blob = torch.zeros(pc.pat_pack_size(F, C, 8, 100, "f16"), dtype=torch.uint8, device="cuda")
    with pytest.raises(pc.PatError) as e:
        pc.pat_pack(torch.zeros((F, C, 3, 3), device="cuda"), torch.full((F, C), 255, dtype=torch.uint8, device="cuda"), masks, 100, "f16", blob=blob)
    assert e.value.code == 2 and not bool(blob.any())
