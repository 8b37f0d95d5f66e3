"""ba_autotune's timing of the defaults is that of the defaults, chunk sizes by
cluster included, and they are the answer where no setting beats them: a
binary64 cluster of some 220 tiles gets chunks of two tiles by default, smaller
than any that can be set, and takes twice as long per linearisation in others."""
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu


def test_defaults_win_where_nothing_beats_them():
    import paper_2511_06152_gb300 as ba
    scene = sg.cluster_c1()
    info = ba.presort_host(scene, ba.BA_FP64)
    assert info["tiles_per_chunk"] == 2
    with ba.Context(precision=ba.BA_FP64, tune_table=None) as ctx:
        default = {k: v for k, v in ctx.get_tune().items() if not k.startswith("ms")}
        t = ctx.autotune([scene], 8)
        assert t["ms_tuned"] == t["ms_default"] > 0
        assert {k: v for k, v in t.items() if not k.startswith("ms")} == default
        assert t["chunk_tiles"] == 0 and ctx.get_tune()["chunk_tiles"] == 0
