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


def test_threads_that_pack_different_sizes():
    """The kernel's shared memory limit belongs to the process: no thread may lower what another one is about to use."""
    import threading
    masks, errors = pc.pat_library_builtin(8), []

    def work(F, C, keep):
        try:
            w = torch.randn((F, C, 3, 3), device="cuda")
            n_keep = int(F * C * keep)
            pid, wm = pc.pat_project(w, masks, n_keep)
            torch.cuda.synchronize()
            stream = torch.cuda.Stream()
            blob = torch.empty(pc.pat_pack_size(F, C, 8, n_keep, "f32"), dtype=torch.uint8, device="cuda")
            for _ in range(60):
                pc.pat_pack(wm, pid, masks, n_keep, "f32", blob=blob, stream=stream)
            stream.synchronize()
            assert torch.equal(pc.pat_unpack(blob, F, C, masks, n_keep, "f32"), wm)
        except Exception as e:                 # shown by the assertion below
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=a) for a in ((32, 39312, 0.1), (3, 38496, 0.25), (32, 38608, 0.05), (5, 39316, 0.5))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
