"""ba_get_state into device memory: written by the export kernel straight to
the caller's arrays, the same bytes as the host read-back, and only the arrays
that were asked for."""
import ctypes

import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("wanted", ["RTX", "X", "RT", "T", ""])
def test_device_state_equals_host_state(precision, wanted):
    import torch

    import paper_2511_06152_gb300 as ba
    scene = sg.tiny_cluster(97, 2, 3, 333)
    with ba.Context(precision=ba.BA_MIXED if precision == "mixed" else ba.BA_FP64) as ctx:
        cid = ctx.create_cluster(scene)
        ctx.run(cid, 3, trace=False)
        host = dict(zip("RTX", ctx.get_state(cid)))
        # one double of offset: aligned for binary64, not for wider stores
        out = {k: torch.full((host[k].size + 1,), -7.0, dtype=torch.float64, device="cuda") for k in "RTX"}
        torch.cuda.synchronize()
        ptr = {k: ctypes.cast(out[k].data_ptr() + 8, ctypes.POINTER(ctypes.c_double)) if k in wanted else None
               for k in "RTX"}
        assert ctx.L.ba_get_state(ctx.h, cid, ptr["R"], ptr["T"], ptr["X"], ba.BA_PTR_DEVICE) == ba.BA_OK
        for k in "RTX":
            got = out[k].cpu().numpy()
            assert got[0] == -7.0
            assert np.array_equal(got[1:], host[k].ravel() if k in wanted else np.full(host[k].size, -7.0))
