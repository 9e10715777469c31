"""The library reduction gives a thread one kernel or two, by the size of the layer."""
import itertools

import pytest
import torch

import paper_2001_07710_b200 as pc
from timing import graph_ms

pytestmark = pytest.mark.gpu

MASKS = [sum(1 << b for b in c) for c in itertools.combinations(range(9), 4)]


def weights(n):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    return torch.randn((n, 3, 3), generator=gen, device="cuda")


@pytest.mark.parametrize("K", [126, 125])
@pytest.mark.parametrize("off", [-257, -1, 0, 1, 256])
def test_counts_next_to_the_line(off, K):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 512 * ((5 * sms + 1) // 2 - 1) + 1 + off          # the line: 2 ceil(n / 512) >= 5 SMs
    w = weights(n)
    bits = torch.tensor([[m >> b & 1 for b in range(9)] for m in MASKS[:K]], dtype=torch.float64, device="cuda")
    best = (w.view(n, 9).double().square() @ bits.T).argmax(1)
    out, counts = pc.pat_extract_library(w, MASKS[:K], 4)
    ref = torch.bincount(best, minlength=K)
    # ties of exact sums aside (none among normal weights), what can differ is a lead of less than the order of fp64 sums gives
    assert int((counts - ref).abs().sum()) <= 2 and int(counts.sum()) == n
    keep = sorted(sorted(range(K), key=lambda j: (-int(counts[j]), j))[:4])
    assert [int(v) & 0xFFFF for v in out] == [MASKS[j] for j in keep]


def test_a_smaller_layer_takes_no_longer():
    """A kernel a thread in a layer of 512 x 512 took half as long again as two: more than a layer of a sixth more kernels."""
    def ms(n):
        w, counts, out = weights(n), torch.empty(126, dtype=torch.int64, device="cuda"), torch.empty(12, dtype=torch.int16, device="cuda")
        return graph_ms(lambda: pc.pat_extract_library(w, MASKS, 12, masks_out=out, counts=counts))
    ms(512 * 512)
    assert ms(512 * 512) <= 1.25 * ms(303105)              # measured 11.8 and 11.0 us; 16.6 and 11.1 with one
