"""An error that a call returned is not returned again by the next one.  The
errors are the host's: calls that a stream capture does not permit, and a launch
on a stream whose capture they ended."""
import ctypes as C
import math

import pytest
import torch

from paper_2401_12724_gb300 import _native as N
from paper_2401_12724_gb300 import api
from paper_2401_12724_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("refused", ["create", "destroy", "trace"])
def test_an_error_is_returned_once(refused):
    lib, cuda = N.load(), C.CDLL("libcuda.so.1")
    M, gone = api.Materials([I.material()]), api.Materials([I.material()])
    params = api.default_params([I.material()]).cuda()
    yarns = api.yarns_to_device(I.woven_scene(1, 1))
    rays = {k: torch.from_numpy(v).cuda() for k, v in I.camera_rays(8, 8, extent=2.5).items()}
    light = (0.3, -0.4, math.sqrt(0.75))
    out = api.trace_yarns(yarns, rays, light)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    arr = (N.MaterialDesc * 1)(api.desc_struct(I.material()))
    handle, graph = C.c_void_p(), C.c_void_p()
    assert cuda.cuStreamBeginCapture_v2(C.c_void_p(st.cuda_stream), 0) == 0  # global
    try:
        if refused == "destroy":
            gone.close()  # synchronises the device; reports nothing
        else:
            # an allocation: refused, and the capture ends with it
            assert lib.bysdf_create_materials(arr, 1, None, C.byref(handle)) == -2
        if refused == "trace":
            with pytest.raises(RuntimeError, match="captur"):
                api.trace_yarns(yarns, rays, light, stream=st, out=out)
    finally:
        cuda.cuStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(graph))
    assert lib.bysdf_set_params(M.handle, params.data_ptr(),
                                torch.cuda.current_stream().cuda_stream) == 0, lib.bysdf_last_error()
    torch.cuda.synchronize()
    assert torch.equal(M.get_params(), params)
