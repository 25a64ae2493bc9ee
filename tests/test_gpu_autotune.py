"""The autotuner's candidates work on every record.  Batches of a few tiles per
warp are where the defaults shorten their tiles; a candidate keeps the tiles of
its own shape, and a tile longer than its kernel's rounds is an error."""
import pytest
import torch

from paper_2401_12724_gb300 import _native as N
from paper_2401_12724_gb300 import api
from paper_2401_12724_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _records(n, sort, ratio):
    rec = I.random_records(n, n_mat=8, seed=81, wi_mode="cosine", ratio=ratio, sample=True,
                           sorted_ids=sort)
    seg = I.seg_offsets_from_ids(rec["mat_id"], 8) if sort else None
    return api.records_to_device(rec, seg_offsets=seg)


# sorted near-field records: 2 rounds per warp, and up to the 16 where the
# defaults' tiles are 2 rounds; footprints: 1, 3 and 9 rounds per warp
@pytest.mark.parametrize("n,sort,ratio", [(150_000, True, None), (300_000, True, None),
                                          (1_100_000, True, None), (300_000, False, None),
                                          (100_000, True, "loguniform"),
                                          (350_000, False, "loguniform"),
                                          (1_000_000, False, "loguniform")])
def test_every_candidate_works_on_every_record(n, sort, ratio):
    M, S = api.Materials(I.materials(2)), api.Materials(I.materials(2))
    d = _records(n, sort, ratio)

    def outputs():
        # no status is 77, lobe included, and no written value either
        o = api.alloc_fused(n, "cuda")
        for v in o.values():
            v.fill_(77)
        return o

    def check_written(o):
        for k, v in o.items():
            assert not (v == 77).any(), k

    for block in (128, 256, 512):
        for items in (1, 2, 4, 8):
            for occ in (0, 1):
                S.set_launch_config(N.OP_FUSED, block, items, occupancy=occ)
                check_written(api.eval_sample_pdf(S, d, out=outputs()))
    o = outputs()
    best = api.autotune(M, N.OP_FUSED, d, out=o)
    check_written(o)
    # the tuned shape is the one that can be set, bit for bit
    S.set_launch_config(N.OP_FUSED, best["block"], best["items"], occupancy=best["occupancy"])
    got, want = api.eval_sample_pdf(M, d, out=outputs()), api.eval_sample_pdf(S, d)
    for k, v in want.items():
        assert torch.equal(v, got[k]), k
    assert M.workspace_error() == 0 and S.workspace_error() == 0
