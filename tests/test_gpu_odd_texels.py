"""Migrating materials whose maps have an odd number of texels: the texels behind
which a migration map's header lies are padded to 16 bytes, in the device table
and in shared memory.  Every kernel that reads it gives the oracle's values."""
import numpy as np
import pytest

import parity_util as PU
from paper_2401_12724_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = 2003


def np_(t):
    return t.detach().cpu().numpy()


# all counts of maps, in any order and as material-sorted slots, from the fewest
# odd texels to nearly the most that 16 slots of two maps hold
@pytest.mark.parametrize("texels,maps,sort", [(5, 2, False), (5, 4, True), (255, 2, False),
                                              (255, 3, True), (257, 4, False), (801, 2, True)])
def test_odd_texel_counts_match_the_oracle(orc, texels, maps, sort):
    from paper_2401_12724_gb300 import api

    mats = I.materials(2)[:2]
    for k, d in enumerate(mats):
        d.update(map_texels=texels, migration_maps=maps, migration_seed=40 + k,
                 migration_length=0.4 + 0.3 * k, migration_blend=0.2)
    rec = I.random_records(N, n_mat=2, seed=texels + maps, wi_mode="cosine", sample=True,
                           sorted_ids=sort, v_max=5.0)
    seg = I.seg_offsets_from_ids(rec["mat_id"], 2) if sort else None
    M = api.Materials(mats)
    d = api.records_to_device(rec, seg_offsets=seg)
    view = PU.oracle_view(orc, lambda r: orc.eval_records(mats, r, threads=8), mats, rec)
    f, p, st = (np_(t) for t in api.eval(M, d))
    PU.assert_status(st, view, "odd")
    PU.assert_parity(f, view, 0, "odd.f", gpu_status=st)
    PU.assert_parity(p, view, 1, "odd.pdf", gpu_status=st)
    for t in (api.sample(M, d), api.eval_stochastic(M, d, 3, 3),
              api.eval_sample_pdf(M, d).values()):
        assert all(torch.isfinite(x).all() for x in t)
    g = np.random.default_rng(96).uniform(-1, 1, (3, N)).astype(np.float32)
    g[:, ~PU.gradient_mask(orc, mats, rec, view)] = 0.0
    want, _, J = orc.grad_records(mats, rec, g.astype(np.float64), threads=8, jac=True)
    scale = np.zeros((2, 8))
    np.add.at(scale, rec["mat_id"], np.abs(g.T[:, :, None] * J).sum(1))
    gt = torch.from_numpy(g).cuda()
    got, gwi, gwo = api.eval_backward_ext(M, d, gt, dirs=True)
    assert torch.isfinite(gwi).all() and torch.isfinite(gwo).all()
    for grad in (api.eval_backward(M, d, gt), got):
        # the tolerance of the parity tests' gradients; the 15 columns split
        # the two body colours, which the 8 move together
        grad = np_(grad).astype(np.float64)
        if grad.shape[1] == 15:
            grad[:, :3] += grad[:, 9:12]
        assert (np.abs(grad[:, :8] - want) <= 1e-4 * scale + 1e-6).all()
    # a parameter update rewrites the headers' rates: setting what was read
    # back changes nothing from then on
    M.set_params(M.get_params())
    a = api.eval(M, d)
    M.set_params(M.get_params())
    b = api.eval(M, d)
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    assert M.workspace_error() == 0
