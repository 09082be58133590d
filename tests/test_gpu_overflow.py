"""Fields past the arithmetic's range: no pose scores above -infinity.

A pocket value is accepted when it is finite in FP32, but -1e5 is -infinity in FP16 cells and the sum of two
lookups of -3e38 is -infinity in FP32, so every pose of a ligand inside such a field scores -infinity or not a
number.  No pose wins then; the choice is pose 0, angle index in range, restart 0, in every form.
"""
import numpy as np
import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,value", [("f16", -1e5), ("f32", -3e38)])
def test_no_pose_above_minus_infinity(grid, value):
    from paper_2209_05069_gb300 import dock
    pk = synth.make_field_pocket((48, 48, 48), 0.5, (-11.75,) * 3, lambda x, y, z: np.full_like(x + y + z, value))
    db = synth.make_db(synth.WORKLOADS["tiny"], 6)
    prm = dock.Params.make(restarts=5, align_steps=9, torsion_steps=40, clash_dist=2.0, seed=3, select_k=2)
    shapes = [None, (4, -1, 0, 1, 2), (4, -1, 1, 1, 1), (8, -1, 0, 2, 1), (4, -1, 0, 4, 1), (8, -1, 0, 8, 1)]
    for form, shape in [(dock.DOCK_FORM_BATCHED, s) for s in shapes] + [(dock.DOCK_FORM_LATENCY, None)]:
        with dock.Context(serve=False) as ctx:
            if shape is not None:
                for b in range(5):
                    ctx.set_launch(b, *shape)
            batch = ctx.batch_create(db, prm)
            ctx.batch_launch(ctx.load(pk, grid), batch, form)
            res = ctx.batch_results(batch)
            ctx.batch_destroy(batch)
        assert not np.isfinite(res["restart_score"]).any()
        assert (res["align_idx"] == 0).all() and (res["post_idx"] == 0).all(), (form, shape)
        assert ((res["torsion_idx"] >= 0) & (res["torsion_idx"] < 40)).all(), (form, shape)
        assert (res["best_restart"] == 0).all() and (res["score"] == -np.inf).all(), (form, shape)
        assert (res["select_restart"].reshape(-1, 2)[:, 0] == 0).all(), (form, shape)
        assert np.isfinite(res["xyz"]).all(), (form, shape)
