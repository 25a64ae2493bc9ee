"""The tiles that the defaults choose by rounds of 32 records per warp: around
every switch a batch gives, record for record, what a larger one gives.
Footprint records switch at 3, 6 and 12 rounds, material-sorted near-field
records at 4 and 16; the stochastic estimators also between two kernels (8)."""
import numpy as np
import pytest
import torch

from paper_2401_12724_gb300 import api
from paper_2401_12724_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _warps(per_sm):
    return per_sm * torch.cuda.get_device_properties(0).multi_processor_count


class Batches:
    """Prefixes of one record set; run(call, n) fills every output first."""

    def __init__(self, top, sort, ratio):
        self.rec = I.random_records(top, n_mat=8, seed=72, wi_mode="cosine", ratio=ratio,
                                    sample=True, sorted_ids=sort)
        self.sort, self.M = sort, api.Materials(I.materials(2))

    def run(self, call, n):
        cut = {k: np.ascontiguousarray(a[..., :n]) for k, a in self.rec.items()}
        seg = I.seg_offsets_from_ids(cut["mat_id"], 8) if self.sort else None
        d = api.records_to_device(cut, seg_offsets=seg)
        o = api.alloc_fused(n, "cuda")
        for v in o.values():
            v.fill_(77)
        call(self.M, d, o)
        torch.cuda.synchronize()
        assert self.M.workspace_error() == 0
        return o

    def check(self, call, sizes, top):
        want = self.run(call, top)
        for n in sizes:
            for k, v in self.run(call, n).items():
                assert torch.equal(v, want[k][..., :n]), (n, k)


def fused(M, d, o):
    api.eval_sample_pdf(M, d, out=o)


def stochastic(M, d, o):
    api.eval_sample_pdf_stochastic(M, d, 11, 3, out=o)


def around(warps, rounds):
    return [32 * warps * r + e for r in rounds for e in (-33, -1, 0, 1, 33)]


@pytest.mark.parametrize("sort", [False, True])
def test_footprint_records(sort):
    # a kernel for each length of tile (1, 2, 4, 8 rounds): bits are compared
    # with the largest batch that takes the same one
    w = _warps(24)
    B = Batches(32 * w * 14 + 5, sort, "loguniform")
    low = 1
    for rounds in (3, 6, 12, 14):
        top = 32 * (w * rounds - 1)  # the last batch below the switch
        B.check(fused, [low, low + 31, low + 33, 32 * w * (rounds - 1) + 7, top - 1], top)
        low = top + 1


def test_sorted_near_field_records():
    w = _warps(20)
    top = 32 * w * 18 + 5
    Batches(top, True, None).check(fused, around(w, (4, 16)), top)


@pytest.mark.parametrize("sort", [False, True])
def test_stochastic_records(sort):
    # footprints: one kernel below 8 rounds a warp, another from there on
    w = _warps(24)
    B = Batches(32 * w * 14 + 5, sort, "loguniform")
    B.check(stochastic, around(w, (3, 6)), 32 * w * 8 - 256)
    B.check(stochastic, around(w, (12,)) + [32 * w * 8], 32 * w * 14 + 5)
    # near-field: tiles of one round below 4 rounds a warp (16 warps)
    w = _warps(16)
    B = Batches(32 * w * 6 + 5, sort, None)
    B.check(stochastic, [1, 33] + around(w, (1, 2)), 32 * w * 4 - 128)
    B.check(stochastic, around(w, (5,)) + [32 * w * 4], 32 * w * 6 + 5)
