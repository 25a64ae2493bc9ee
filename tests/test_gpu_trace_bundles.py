"""A ray's result does not depend on the rays it shares a warp with: traced in
row order (tight bundles, some of them over a row's end) and in a shuffled
order (bundles that keep most pieces), every output has the same bits."""
import math

import numpy as np
import pytest
import torch

from paper_2401_12724_gb300 import api
from paper_2401_12724_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LIGHT = (0.3, -0.4, math.sqrt(0.75))


# below and above one large CTA per SM (152 x 768 rays); widths that are a
# multiple of the warp and not; pieces at the edges of a group of 8, of 32
# groups and at the most that is taken
@pytest.mark.parametrize("w,h", [(1, 1), (33, 7), (96, 80), (333, 351), (512, 256)])
@pytest.mark.parametrize("n_yarns,pieces,keep", [(1, 1, 1), (3, 3, 17), (9, 15, 257), (32, 32, 2048)])
def test_rays_do_not_depend_on_their_neighbours(w, h, n_yarns, pieces, keep):
    scene = I.woven_scene(n_yarns, pieces)[:keep]
    rays = I.camera_rays(w, h, extent=pieces * 2.5, jitter_seed=3)
    order = np.random.default_rng(w * h + keep).permutation(w * h)
    yarns = api.yarns_to_device(scene)

    def trace(perm):
        r = {k: torch.from_numpy(np.ascontiguousarray(v[:, perm])).cuda() for k, v in rays.items()}
        return api.trace_yarns(yarns, r, LIGHT)

    want, got = trace(np.arange(w * h)), trace(order)
    idx = torch.from_numpy(order).cuda()
    for k, v in want.items():
        assert torch.equal(v[..., idx], got[k]), k
