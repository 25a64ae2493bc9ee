"""Every record of a batch is worked on once, whatever the tiles: sizes around
one round per warp, the switch from short to full tiles and the last partial
tile give, record for record, what one large batch gives."""
import numpy as np
import pytest
import torch

from paper_2401_12724_gb300 import api
from paper_2401_12724_gb300 import inputs as I

pytestmark = pytest.mark.gpu
WARPS = 152 * 20  # resident warps of the near-field shape on 152 SMs


def _outputs(M, d, n):
    o = api.alloc_fused(n, "cuda")
    for v in o.values():
        v.fill_(77)
    return api.eval_sample_pdf(M, d, out=o)


@pytest.mark.parametrize("ratio", [None, "loguniform"])
@pytest.mark.parametrize("sort", [False, True])
def test_batches_around_tile_edges(ratio, sort):
    top = 32 * WARPS * 6 + 77 if ratio is None else 32 * 3648 * 4 + 77
    rec = I.random_records(top, n_mat=8, seed=71, wi_mode="cosine", ratio=ratio, sample=True,
                           sorted_ids=sort)
    M = api.Materials(I.materials(2))

    def run(n):
        cut = {k: np.ascontiguousarray(a[..., :n]) for k, a in rec.items()}
        seg = I.seg_offsets_from_ids(cut["mat_id"], 8) if sort else None
        return _outputs(M, api.records_to_device(cut, seg_offsets=seg), n)

    want = {k: v.clone() for k, v in run(top).items()}
    sizes = [1, 31, 32, 33, 32 * WARPS - 1, 32 * WARPS, 32 * WARPS + 1, 32 * WARPS * 4,
             32 * WARPS * 4 + 33, 32 * WARPS * 5 - 5]
    for n in [s for s in sizes if s <= top]:
        got = run(n)
        torch.cuda.synchronize()
        assert M.workspace_error() == 0
        for k, v in got.items():
            assert torch.equal(v, want[k][..., :n]), (n, k)
