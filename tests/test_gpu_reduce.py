"""The sums of the chunk partials of an image or image pair, at list lengths
around the split of a list into runs (six runs, eight rows in flight): one
chunk, a few, and hundreds.  FP64 steps against the oracle at the parity
tolerance; in mixed precision, the same cluster's first step against the
binary64 path's within its binary32 rounding."""
import numpy as np
import pytest

import oracle as O
import scenegen as sg
from helpers import fp64_step_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("points", [24, 200, 380, 420, 2600, 3300, 20000])
def test_partial_sums_of_any_list_length(points):
    import paper_2511_06152_gb300 as ba
    scene = sg.tiny_cluster(1000 + points, 1, 4, points, fixed=(0,))
    assert fp64_step_parity(ba, O, scene, 2) == 2
    state = {}
    for prec in (ba.BA_FP64, ba.BA_MIXED):
        with ba.Context(precision=prec) as ctx:
            cid = ctx.create_cluster(scene)
            assert ctx.run(cid, 1)[0]["accepted"] == 1
            state[prec] = ctx.get_state(cid)
    # the centres' corrections (0.05 m) carry the binary32 rounding of the
    # observations' residuals (about 5e-4 px of 0.5 px) and nothing larger
    d = np.abs(state[ba.BA_MIXED][1] - state[ba.BA_FP64][1]).max()
    assert d < 1e-3 * 0.05 * 3, d
