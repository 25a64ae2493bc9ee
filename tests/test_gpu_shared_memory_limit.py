"""Launches around 48 KB of shared memory.  A kernel may use 48 KB of static
plus dynamic shared memory before its limit is raised, so sizes whose dynamic
part alone stays below 48 KB need the raise as well.  The limit is raised for
the rest of the process: each test runs in a process of its own and goes
through the sizes in ascending order, so that no earlier call has raised it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _child(body):
    code = "import math\nimport numpy as np\nimport torch\n" \
           "from paper_2401_12724_gb300 import api\n" \
           "from paper_2401_12724_gb300 import inputs as I\n" + body
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]


# 68 bytes a piece and 16 a group of 8: 702 pieces are 49,144 bytes, with
# 256 (CTAs of 256 threads) or 768 bytes (of 768) of static lists on top
TRACE = """
near = I.woven_scene(5, 5)[:40]
far = [dict(near[0], p0=[500.0 + 3.0 * k, 400.0, -300.0]) for k in range(710)]
w, h = {shape}
rays = {{k: torch.from_numpy(v).cuda()
        for k, v in I.camera_rays(w, h, extent=12.5, jitter_seed=3).items()}}
light = (0.3, -0.4, math.sqrt(0.75))
want = api.trace_yarns(api.yarns_to_device(near), rays, light)
assert (want["yarn_id"] >= 0).any()
for n in (680, 691, 692, 696, 699, 700, 702, 703, 704, 720):
    got = api.trace_yarns(api.yarns_to_device(near + far[: n - 40]), rays, light)
    for k, v in want.items():
        assert torch.equal(v, got[k]), (n, k)
"""


# one 768-thread CTA per SM takes 152 x 768 rays, fewer go in CTAs of 256
@pytest.mark.parametrize("shape", [(96, 80), (512, 256)])
def test_traces_of_690_to_720_pieces(shape):
    _child(TRACE.format(shape=shape))
