"""Torsion sweeps of up to 32 angles with 8 warps per item (a bump check of one pass) choose as every other shape does:
angle counts around a single pass, thresholds from none to most of a molecule, in batches and in the latency form."""
import numpy as np
import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu


def _db():
    ligs = []
    for i, n in enumerate([9, 32, 33, 64, 96, 97, 160]):
        rng = np.random.Generator(np.random.PCG64([78, n]))
        xyz, bonds, rot, _ = synth.make_ligand(rng, n, min(6, n // 6))
        ligs.append((xyz, bonds, rot, i))
    return synth.from_ligands(ligs)


@pytest.mark.parametrize("grid", ["f32", "i16"])
@pytest.mark.parametrize("angles", [1, 2, 31, 32, 33])
def test_one_pass_bump_check(angles, grid):
    from paper_2209_05069_gb300 import dock
    pk, db = synth.workload_pocket(synth.WORKLOADS["tiny"]), _db()
    if grid == "i16":
        pk = pk.integer(1000)
    for clash in (0.0, 2.0, 9.0):
        for early in (0, 1):
            prm = dock.Params.make(restarts=3, align_steps=6, torsion_steps=angles, clash_dist=clash, seed=2, early_exit=early)
            runs = []
            for shape, form in (((4, -1, 0, 1, 1), 0), ((8, -1, 0, 8, 1), 0), (None, dock.DOCK_FORM_LATENCY)):
                with dock.Context(serve=False) as ctx:
                    if shape is not None:
                        for b in range(5):
                            ctx.set_launch(b, *shape)
                    batch = ctx.batch_create(db, prm)
                    ctx.batch_launch(ctx.load(pk, grid), batch, form)
                    runs.append(ctx.batch_results(batch))
                    ctx.batch_destroy(batch)
            for other in runs[1:]:
                for k in runs[0]:
                    assert np.array_equal(runs[0][k], other[k]), (k, clash, early)
