"""Observations whose weight is zero in the mixed path's back-substitution:
points far off to the side and behind the images that observe them.  They add
nothing to a step, as in binary64, however large their coordinates are."""
import numpy as np
import pytest

import scenegen as sg
from helpers import rms_inliers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("far", [1e3, 1e5, 4e6])
def test_points_behind_images_leave_the_steps_alone(far):
    import paper_2511_06152_gb300 as ba
    c = sg.tiny_cluster(77, 2, 3, 400)
    c = {key: (v.copy() if isinstance(v, np.ndarray) else v) for key, v in c.items()}
    c["intr"][:, 3:7] = 1e-3
    # one more point, above and far beside the images, observed by half of them;
    # at that height it lies behind every image whatever its tilt of half a degree
    j, seen_by = int(c["n_pts"]), np.arange(0, 6, 2)
    c["X0"] = np.vstack([c["X0"], [[far, 0.3 * far, 300.0 + 0.2 * far]]])
    c["obs_cam"] = np.concatenate([c["obs_cam"], seen_by.astype(np.int32)])
    c["obs_pt"] = np.concatenate([c["obs_pt"], np.full(3, j, np.int32)])
    c["obs_uv"] = np.vstack([c["obs_uv"], np.tile([4000.0, 3000.0], (3, 1))])
    c["n_pts"], c["n_obs"] = j + 1, int(c["n_obs"]) + 3
    out = {}
    for prec in (ba.BA_FP64, ba.BA_MIXED):
        with ba.Context(precision=prec) as ctx:
            cid = ctx.create_cluster(c)
            out[prec] = ctx.run(cid, 4), ctx.get_state(cid)
            rms = rms_inliers(ctx.reprojection_errors(cid)[:-3], c["outlier"])
            out[prec] += (rms,)
    ref, got = out[ba.BA_FP64], out[ba.BA_MIXED]
    # the decisions; the mixed path's parity bounds (1 mm, 1e-3 px); the far point stays where it is
    assert all(a["accepted"] == b["accepted"] == 1 for a, b in zip(got[0][:3], ref[0][:3]))
    assert sg.centre_error(got[1][1], ref[1][1]) < 1e-3
    assert abs(got[2] - ref[2]) < 1e-3
    assert np.array_equal(got[1][2][j], c["X0"][j])
