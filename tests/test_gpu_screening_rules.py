"""Which launches screen their alignments, seen by the counter build: estimates are loads that are not lookups, so a
launch that screens issues more loads than lookups and looks up few of its poses; one that does not issues at most
one load per lookup.  Results of both are compared bit for bit with every pose scored in test_gpu_screening.py."""
import numpy as np
import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu

ONE, TWO, FOUR, EIGHT = (4, -1, 0, 1, 2), (8, -1, 0, 2, 1), (8, -1, 0, 4, 1), (8, -1, 0, 8, 1)


def _work(grid, shape, db, pk, **params):
    from paper_2209_05069_gb300 import dock
    with dock.Context(serve=False, counters=True) as ctx:
        if shape is not None:
            for b in range(5):
                ctx.set_launch(b, *shape)
        prm = dock.Params.make(**dict(dict(restarts=10, align_steps=30, torsion_steps=32, seed=3), **params))
        b = ctx.batch_create(db, prm)
        ctx.batch_launch(ctx.load(pk, grid), b)
        ctx.batch_wait(b)
        work, algo = ctx.exec_counters(), ctx.batch_work(b)
        ctx.batch_destroy(b)
    return work, algo


def _screened(work, algo):
    """Whether the alignments were screened; every launch here is all or nothing."""
    if work["loads"] > work["lookups"]:
        assert work["lookups"] - algo["lookups_torsion"] - algo["lookups_final"] < 0.25 * algo["lookups_align"]
        return True
    assert work["lookups"] > algo["lookups_align"]
    return False


@pytest.mark.parametrize("grid,shape,steps,screened", [
    ("f32", ONE, 16, True), ("f32", ONE, 15, False), ("f32", TWO, 18, True), ("f32", TWO, 17, False),
    ("f32", FOUR, 22, True), ("f32", FOUR, 21, False), ("f32", EIGHT, 30, False), ("f32", ONE, 6, False),
    ("f16", ONE, 20, True), ("f16", ONE, 19, False), ("f16", TWO, 24, True), ("f16", TWO, 23, False),
    ("f16", FOUR, 30, False), ("f32", TWO, 64, True), ("f16", TWO, 128, True), ("f32", FOUR, 128, True)])
def test_poses_per_warp(grid, shape, steps, screened):
    w = synth.WORKLOADS["tiny"]
    db = synth.make_db(w, 4 if steps > 60 else 40)
    assert _screened(*_work(grid, shape, db, synth.workload_pocket(w), align_steps=steps)) == screened


def _sized(n_atoms, count):
    ligs = []
    for i in range(8):
        rng = np.random.Generator(np.random.PCG64([9, n_atoms, i]))
        xyz, bonds, rot, _ = synth.make_ligand(rng, n_atoms, 3)
        ligs.append((xyz, bonds, rot, i))
    return synth.tile_db(synth.from_ligands(ligs), count)


@pytest.mark.parametrize("grid,shape,atoms,ligands,screened", [
    # 28 warps per SM of 152: 4,256 one-warp items, 2,128 of two warps; with 4 warps 40: 1,520
    ("f32", ONE, 110, 430, True), ("f32", ONE, 110, 420, False), ("f32", TWO, 110, 215, True), ("f32", TWO, 110, 210, False),
    ("f32", FOUR, 110, 155, True), ("f32", FOUR, 110, 150, False),
    # up to 96 atoms 8 with 1 and 4 warps: 1,216 and 304 items, none with 2
    ("f32", ONE, 90, 125, True), ("f32", ONE, 90, 118, False), ("f32", FOUR, 90, 32, True), ("f32", FOUR, 90, 29, False),
    ("f16", ONE, 90, 118, False), ("f16", TWO, 90, 4, True), ("f32", ONE, 60, 4, True),
    ("f16", TWO, 110, 215, True), ("f16", TWO, 110, 210, False), ("f16", ONE, 110, 430, True), ("f16", ONE, 110, 420, False)])
def test_large_molecules_need_a_full_gpu(grid, shape, atoms, ligands, screened):
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes are those of 152 SMs")
    pk = synth.workload_pocket(synth.WORKLOADS["uneven"])
    assert _screened(*_work(grid, shape, _sized(atoms, ligands), pk, torsion_steps=8)) == screened
