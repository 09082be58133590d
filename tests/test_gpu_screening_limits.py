"""Fields that screening does not suit: a launch gives up soon, seen by the counter build.

Every atom stays where voxels are not zero, so each lookup issues one load and the loads beyond them are estimates.
Results on such fields are compared bit for bit with every pose scored in test_gpu_screening.py."""
import dataclasses

import numpy as np
import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu


def _field(name):
    """A box of constant value with zero faces, around which nothing of a 20-30 atom ligand reaches."""
    def box(x, y, z):
        return np.where(np.maximum(np.maximum(abs(x), abs(y)), abs(z)) < 17.9, 1.0, 0.0)
    pk = synth.make_field_pocket((73, 73, 73), 0.5, (-18.0,) * 3, box)
    if name == "walls":       # a few deep voxels: their range hides the differences between poses
        v = pk.values.copy()
        rng = np.random.Generator(np.random.PCG64(5))
        v += (0.1 * rng.random(v.shape) * (v > 0)).astype(np.float32)
        v[(rng.random(v.shape) < 0.002) & (v > 0)] = -5000.0
        return dataclasses.replace(pk, values=np.ascontiguousarray(v, np.float32))
    if name == "constant":    # small variation on a large constant
        return synth.make_field_pocket((73, 73, 73), 0.5, (-18.0,) * 3,
                                       lambda x, y, z: 500.0 + np.sin(2.0 * x) + np.cos(1.7 * y + z))
    return pk


def _estimates(field, grid, ligands, steps=20):
    """Estimates made, and the ligands' lookups of one pose in one alignment."""
    from paper_2209_05069_gb300 import dock
    db = synth.tile_db(synth.make_db(synth.WORKLOADS["tiny"], 32), ligands)
    prm = dock.Params.make(restarts=30, align_steps=steps, torsion_steps=8, seed=3)
    with dock.Context(serve=False, counters=True) as ctx:
        for b in range(5):
            ctx.set_launch(b, 4, -1, 0, 1, 2)
        b = ctx.batch_create(db, prm)
        ctx.batch_launch(ctx.load(_field(field), grid), b)
        ctx.batch_wait(b)
        work = ctx.exec_counters()
        ctx.batch_destroy(b)
    assert work["lookups"] >= 0.99 * 2 * steps * steps * 30 * int(db.atom_off[-1]), "an alignment was screened to the end"
    return work["loads"] - work["lookups"], 30 * int(db.atom_off[-1])


@pytest.mark.parametrize("grid", ["f32", "f16"])
@pytest.mark.parametrize("field", ["flat", "walls"])
@pytest.mark.parametrize("ligands,alignments", [(100, 2), (700, 1)])   # below and above 100 ligand-restarts per SM
def test_giving_up(field, grid, ligands, alignments):
    """One block of 64 poses is estimated (in the walls' field up to three, in some alignments), in the first alignment
    alone where the launch fills the GPU many times over."""
    estimates, pose = _estimates(field, grid, ligands)
    assert 0 < estimates <= alignments * (64 if field == "flat" else 3 * 64) * pose


@pytest.mark.parametrize("grid", ["f32", "f16"])
def test_a_large_constant_is_not_screened(grid):
    assert _estimates("constant", grid, 100)[0] == 0
