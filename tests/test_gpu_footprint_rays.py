"""A warp per footprint ray: rays of a single sample (flat ground), of fewer
than 32, of several hundred (oblique rays over a fine raster), rays that do
not point down, and rasters that are refused."""
import numpy as np
import pytest
from scipy.spatial.transform import Rotation

import oracle as O
import scenegen as sg

pytestmark = pytest.mark.gpu

W, H, F = sg.SENSOR_W, sg.SENSOR_H, sg.FOCAL_PX


def _raster(seed, cell, relief):
    rng = np.random.Generator(np.random.PCG64(seed))
    x = cell * np.arange(int(240 / cell))
    y = cell * np.arange(int(200 / cell))
    h = relief * (np.sin(x[None, :] / 17.0) + np.cos(y[:, None] / 23.0)) + 0.1 * relief * rng.random((len(y), len(x)))
    return dict(h=h, x0=-120.0, y0=-100.0, dx=cell, dy=cell)


@pytest.mark.parametrize("cell,relief,tilt", [(2.0, 0.0, 0.0), (5.0, 4.0, 2.0), (1.0, 12.0, 25.0), (0.5, 20.0, 55.0),
                                              (2.0, 10.0, 80.0)])
@pytest.mark.parametrize("n", [1, 33])
def test_rays_match_oracle(cell, relief, tilt, n):
    import paper_2511_06152_gb300 as ba
    dsm = _raster(int(10 * cell) + n, cell, relief)
    rng = np.random.Generator(np.random.PCG64(n))
    R = np.stack([sg.nadir_rotation(rng.uniform(0, 6.28)) @ Rotation.from_euler("x", tilt, degrees=True).as_matrix()
                  for _ in range(n)])
    T = np.column_stack([rng.uniform(-60, 60, n), rng.uniform(-60, 60, n), np.full(n, 150.0)])
    intr = np.tile([F, W / 2, H / 2, 0, 0, 0, 0], (n, 1))
    with ba.Context() as ctx:
        q = ctx.footprints(intr, W, H, R, T, dsm)
    D = O.Dsm(dsm)
    for k in range(n):
        ref = O.footprint(intr[k], W, H, R[k], T[k], D)
        if ref is None:
            assert np.isnan(q[k]).any()
        else:
            np.testing.assert_allclose(q[k], ref, atol=1e-6)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_raster_is_refused(bad):
    import paper_2511_06152_gb300 as ba
    dsm = _raster(3, 2.0, 5.0)
    dsm["h"][7, 11] = bad
    intr = np.array([[F, W / 2, H / 2, 0, 0, 0, 0]])
    with ba.Context() as ctx:
        with pytest.raises(ba.BAError) as e:
            ctx.footprints(intr, W, H, sg.nadir_rotation(0.0)[None], np.array([[0.0, 0.0, 150.0]]), dsm)
        assert e.value.status == ba.BA_ERR_INVALID
