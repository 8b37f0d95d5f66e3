"""The LM step taken at the end of the back-substitution's CTAs: batches in
which a CTA completes no cluster, a few, and more than its list holds (72 of
one-tile clusters, on a grid of one CTA per SM), each cluster's result equal
bit for bit to the one it gets alone."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,clusters", [("mixed", 3), ("mixed", 200), ("mixed", 9800), ("fp64", 9800)])
def test_lm_steps_of_many_small_clusters(precision, clusters):
    import paper_2511_06152_gb300 as ba
    scenes = [sg.tiny_cluster(60 + i, 1, 3, 9) for i in range(3)]
    with ba.Context(precision=ba.BA_MIXED if precision == "mixed" else ba.BA_FP64) as ctx:
        ctx.set_tune(back_ctas_per_sm=1)
        alone = []
        for sc in scenes:
            cid = ctx.create_cluster(sc)
            ctx.run(cid, 4, trace=False)
            alone.append(ctx.get_state(cid))
        ids = [ctx.create_cluster(scenes[i % 3]) for i in range(clusters)]
        res = ctx.solve_batch(ids, 4)
        assert all(r["status"] == 0 for r in res)
        assert all(res[i]["final_cost"] == res[i % 3]["final_cost"] for i in range(clusters))
        for i, got in enumerate(ctx.get_state_batch(ids)):
            assert all(np.array_equal(a, b) for a, b in zip(got, alone[i % 3]))
