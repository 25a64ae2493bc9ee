"""The autotuner's candidates work on every record.  Batches of a few tiles per
warp are where the defaults shorten their tiles; a candidate keeps the tiles of
its own shape, and a tile longer than its kernel's rounds is an error."""
import ctypes as C

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
    # what is in use is the shape that is reported, or the defaults, bit for bit
    S.set_launch_config(N.OP_FUSED, best["block"], best["items"], occupancy=best["occupancy"])
    D = api.Materials(I.materials(2))
    got = api.eval_sample_pdf(M, d, out=outputs())
    in_use = [S] + ([D] if best == D.launch_config(N.OP_FUSED) else [])
    wants = [api.eval_sample_pdf(X, d) for X in in_use]
    assert any(all(torch.equal(v, got[k]) for k, v in w.items()) for w in wants)
    assert M.workspace_error() == 0 and S.workspace_error() == 0


class _KernelNode(C.Structure):
    """CUDA_KERNEL_NODE_PARAMS (v2) of the driver API."""
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3),
                ("smem", C.c_uint), ("params", C.c_void_p), ("extra", C.c_void_p),
                ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def _launched_blocks(call):
    """Threads per CTA of the kernels that call(stream) launches, from a capture."""
    cuda = C.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph, count = C.c_void_p(), C.c_size_t()
    assert cuda.cuStreamBeginCapture_v2(C.c_void_p(st.cuda_stream), 2) == 0  # relaxed
    try:
        call(st)
    finally:
        rc = cuda.cuStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(graph))
    assert rc == 0
    assert cuda.cuGraphGetNodes(graph, None, C.byref(count)) == 0
    nodes = (C.c_void_p * count.value)()
    assert cuda.cuGraphGetNodes(graph, nodes, C.byref(count)) == 0
    blocks = []
    for node in nodes:
        kind, k = C.c_int(), _KernelNode()
        assert cuda.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)) == 0
        if kind.value == 0:  # a kernel
            assert cuda.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(k)) == 0
            blocks.append(k.block[0])
    assert cuda.cuGraphDestroy(graph) == 0
    return blocks


def test_the_defaults_are_a_candidate_and_can_be_restored():
    M = api.Materials(I.materials(2))
    d = _records(1 << 22, False, None)
    o = api.alloc_fused(1 << 22, "cuda")

    def call(st=None):
        return api.eval_sample_pdf(M, d, out=o, stream=st)

    call()
    assert _launched_blocks(call) == [640]
    M.set_launch_config(N.OP_FUSED, 128, 2)
    call()
    assert _launched_blocks(call) == [128]
    # on these records the defaults are 3% faster than any shape that can be
    # set, and come back into use with their tile rules
    assert api.autotune(M, N.OP_FUSED, d, out=o) == M.launch_config(N.OP_FUSED)
    assert _launched_blocks(call) == [640]
    M.set_launch_config(N.OP_FUSED, 128, 2)
    M.reset_launch_config(N.OP_FUSED)
    assert _launched_blocks(call) == [640]
    assert M.launch_config(N.OP_FUSED) == api.Materials(I.materials(2)).launch_config(N.OP_FUSED)
    with pytest.raises(RuntimeError):
        M.reset_launch_config(5)
    M.reset_launch_config(N.OP_BACKWARD)
    assert M.launch_config(N.OP_BACKWARD)["items"] == 8
