"""The tensor-core solver over the scale of its system: with every sigma
smaller by a power of two the whole problem grows by one, every operation is
exact in that factor, and the steps are the same bits, as long as the system
itself lies inside the binary32 exponent range."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("log2", [8, 20, 26])
def test_steps_do_not_depend_on_the_scale_of_the_sigmas(precision, log2):
    import paper_2511_06152_gb300 as ba
    out = []
    for s in (1.0, 2.0 ** -log2):
        c = sg.tiny_cluster(5151, 4, 10, 3000, fixed=(0, 11))
        for key in ("sigma_px", "sigma_gnss", "sigma_imu"):
            c[key] = c[key] * s
        with ba.Context(precision=ba.BA_FP64 if precision == "fp64" else ba.BA_MIXED) as ctx:
            cid = ctx.create_cluster(c)
            assert ctx.cluster_info(cid)["n_free"] > 32
            steps = ctx.run(cid, 3)
            assert all(x["status"] == 0 for x in steps)
            out.append(([x["accepted"] for x in steps], [x["F_after"] * s * s for x in steps], ctx.get_state(cid)))
    assert out[0][0] == out[1][0] == [1, 1, 1]
    assert out[0][1] == out[1][1]
    for a, b in zip(out[0][2], out[1][2]):
        assert np.array_equal(a, b)
