"""Free images that observe nothing, in a context that has solved and destroyed
other clusters: their sums are zero whatever the memory held before, and the
steps match the oracle as in a fresh context."""
import numpy as np
import pytest

import oracle as O
import scenegen as sg
from helpers import compare_steps, state_rel_err

pytestmark = pytest.mark.gpu


def _with_unobserved_image(c):
    """The scene with one more free image, a copy of image 2 without
    observations, whose pose starts off its priors."""
    c = {key: (v.copy() if isinstance(v, np.ndarray) else v) for key, v in c.items()}
    nc = int(c["n_cams"])
    for key in ("intr", "R0", "T0", "R_prior", "T_prior", "R_true", "T_true", "fixed", "strip"):
        c[key] = np.concatenate([c[key], c[key][2:3]], axis=0)
    c["T0"][nc] += (0.3, -0.2, 0.1)
    c["n_cams"] = nc + 1
    return c


def _without_observations(c):
    c = {key: (v.copy() if isinstance(v, np.ndarray) else v) for key, v in c.items()}
    c["T0"] += (0.3, -0.2, 0.1)
    c.update(n_pts=0, n_obs=0, X0=np.zeros((0, 3)), obs_cam=np.zeros(0, np.int32), obs_pt=np.zeros(0, np.int32),
             obs_uv=np.zeros((0, 2)), outlier=np.zeros(0, bool))
    return c


# up to 32 free images (the shared-memory factor) and more (the global-memory solver)
@pytest.mark.parametrize("strips,per,points", [(2, 3, 200), (4, 10, 3000)])
@pytest.mark.parametrize("kind", ["one image", "all images"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_unobserved_images_after_other_clusters(strips, per, points, kind, precision):
    import paper_2511_06152_gb300 as ba
    seen = sg.tiny_cluster(41, strips, per, points)
    scene = _with_unobserved_image(seen) if kind == "one image" else _without_observations(seen)
    P, S = O.Problem(scene), O.State(scene)
    with ba.Context(precision=ba.BA_FP64 if precision == "fp64" else ba.BA_MIXED) as ctx:
        for n in (points, 4 * points, 2 * points):  # sizes around the scene's: its memory has held their sums
            old = ctx.create_cluster(sg.tiny_cluster(n, strips, per, n))
            ctx.run(old, 2, trace=False)
            ctx.destroy_cluster(old)
        cid = ctx.create_cluster(scene)
        if precision == "fp64":
            assert compare_steps(ctx, cid, O, P, S, 4) >= 2
        else:
            steps = ctx.run(cid, 4)
            for s in steps:
                ref = O.lm_step(P, S)
                assert s["status"] == 0 and s["accepted"] == ref["accepted"]
            R, T, X = ctx.get_state(cid)
            # the unobserved image's pose depends on its priors alone; the others carry binary32 rounding
            if kind == "one image":
                assert np.abs(T[-1] - S.T[-1]).max() < 1e-6 and np.abs(R[-1] - S.R[-1]).max() < 1e-8
                assert sg.centre_error(T, S.T) < 1e-3
            else:
                assert state_rel_err(R, T, X, S.R, S.T, S.X) < 1e-6
