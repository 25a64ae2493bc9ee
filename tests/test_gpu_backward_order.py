"""Gradients of records in any material order: the warp lists a tile's records
by material and folds a material's lanes into one sum, so the sizes where the
list, the rounds or the buckets end are checked against the deterministic
material-sorted pass over the same records."""
import numpy as np
import pytest
import torch

from paper_2401_12724_gb300 import api
from paper_2401_12724_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _materials(n_mat, texels):
    g = np.random.Generator(np.random.Philox(key=[77, n_mat]))
    return [I.material(n_plies=int(g.integers(2, 6)), map_texels=texels,
                       beta_deg=[float(np.float32(g.uniform(5, 20)))] * 2,
                       albedo=[float(np.float32(a)) for a in g.uniform(0.1, 0.9, 3)])
            for _ in range(n_mat)]


# 2 and 20 materials: one bucket each; 33 and 150: several materials a bucket
@pytest.mark.parametrize("n_mat,texels", [(2, 256), (20, 256), (33, 4), (150, 4)])
@pytest.mark.parametrize("n", [1, 31, 33, 511, 513, 20011])
def test_any_order_sums_equal_sorted_sums(n, n_mat, texels):
    import oracle

    mats = _materials(n_mat, texels)
    rec = I.random_records(n, n_mat=n_mat, seed=900 + n, wi_mode="cosine", v_max=5.0)
    rec["mat_id"][: n // 3] = rec["mat_id"][0]  # a run of one material, then all
    if n > 40:
        rec["mat_id"][7] = n_mat  # out of range: contributes nothing
    order = np.argsort(rec["mat_id"], kind="stable")
    srt = {k: np.ascontiguousarray(a[..., order]) for k, a in rec.items()}
    seg = I.seg_offsets_from_ids(np.minimum(srt["mat_id"], n_mat), n_mat + 1)[: n_mat + 1]
    g = np.random.Generator(np.random.Philox(key=[78, n])).uniform(-1, 1, (3, n)).astype(np.float32)
    M = api.Materials(mats)
    d = api.records_to_device(rec)
    got = api.eval_backward(M, d, torch.from_numpy(g).cuda())
    m_last = int(seg[-1])
    keep = {k: np.ascontiguousarray(a[..., :m_last]) for k, a in srt.items()}
    ds = api.records_to_device(keep, seg_offsets=seg)
    gs = torch.from_numpy(np.ascontiguousarray(g[:, order][:, :m_last])).cuda()
    want = api.eval_backward(M, ds, gs, deterministic=True)
    torch.cuda.synchronize()
    assert M.workspace_error() == 0
    # the two add the same numbers in another order: each sum of k terms is
    # within k 2^-24 of the sum of their magnitudes
    _, _, J = oracle.grad_records(mats, keep, gs.cpu().numpy(), threads=4, jac=True)
    mag = np.abs(np.einsum("cn,ncp->np", gs.cpu().numpy().astype(np.float64), J))
    for m in range(n_mat):
        part = mag[seg[m]:seg[m + 1]]
        tol = 2.0 * max(len(part), 1) * 2.0 ** -24 * part.sum(0) * 2.0 + 1e-30
        err = np.abs(got[m].cpu().numpy().astype(np.float64) - want[m].cpu().numpy())
        assert (err <= tol).all(), (m, err, tol)
