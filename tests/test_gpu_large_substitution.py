"""The global-memory solver's substitutions at the orders where their 32-row
block columns, dealt out to the CTAs of a cluster in turn, can go wrong: fewer
block columns than CTAs, exactly full ones, a last block of six rows, a narrow
band (one strip) and a nearly dense envelope (four), fixed images in between;
the double-float factor's step against the binary64 factor's, without and with
refinement passes."""
import pytest

import scenegen as sg
from helpers import state_rel_err

pytestmark = pytest.mark.gpu

# strips, images per strip, fixed images: n = 198 .. 576
SIZES = [(1, 34, 1), (3, 11, 0), (1, 43, 0), (4, 12, 0), (2, 27, 1), (1, 65, 1), (4, 24, 0)]


@pytest.mark.parametrize("strips,per,n_fixed", SIZES)
@pytest.mark.parametrize("refine", [0, 2])
def test_factors_agree(strips, per, n_fixed, refine):
    import paper_2511_06152_gb300 as ba
    scene, out = sg.tiny_cluster(9 * strips + per, strips, per, 50 * strips * per, fixed=range(n_fixed)), {}
    for flags in (0, ba.BA_FLAG_BIG_FP64_FACTOR):
        with ba.Context(precision=ba.BA_FP64, flags=flags, refine_steps=refine) as ctx:
            cid = ctx.create_cluster(scene)
            assert ctx.run(cid, 1)[0]["status"] == 0
            out[flags] = ctx.get_state(cid)
    # double-float rounding (2^-46) times the condition (below 1e7 for the
    # longest strips with the priors on), on steps below a metre
    assert state_rel_err(*out[0], *out[ba.BA_FLAG_BIG_FP64_FACTOR]) < (2e-7 if refine == 0 else 1e-10)
