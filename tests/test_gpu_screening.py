"""The alignment's screening (early_exit on a trilinear grid) and the launch shapes chosen by batch size
change no result.

Scoring every pose in full is the reference (early_exit=0; the oracle checks that path elsewhere): every
output has to be equal bit for bit.  The fields and sizes are those where screening can go wrong: voxels at
the grid's faces that are not zero, fields flat to within the estimates' bound, ligands that reach past the
padded grid, values far from 0 or of large range, rotation counts around a warp's and a pass's width.
"""
import dataclasses

import numpy as np
import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dk():
    from paper_2209_05069_gb300 import dock
    return dock


def _run(dk, pk, grid, db, prm, shape=None):
    with dk.Context(serve=False) as ctx:
        if shape is not None:
            for b in range(5):
                ctx.set_launch(b, *shape)
        b = ctx.batch_create(db, prm)
        ctx.batch_launch(ctx.load(pk, grid), b)
        ctx.batch_wait(b)
        res = ctx.batch_results(b)
        ctx.batch_destroy(b)
    return res


def _same(a, b, what):
    for k in a:
        assert np.array_equal(a[k], b[k]), (what, k)


def _mixed(n_each=2):
    """Ligands of every atom bucket, from the smallest to the largest."""
    ligs = []
    for i, n in enumerate([2, 9, 31, 32, 33, 64, 65, 96, 97, 128, 129, 160]):
        for r in range(n_each):
            rng = np.random.Generator(np.random.PCG64([77, n, r]))
            xyz, bonds, rot, _ = synth.make_ligand(rng, n, min(6, n // 6))
            ligs.append((xyz, bonds, rot, 1000 * i + r))
    return synth.from_ligands(ligs)


def _field(name):
    w = synth.WORKLOADS["tiny"]
    base = synth.workload_pocket(w)
    if name == "workload":
        return base
    if name == "faces":      # nonzero everywhere, faces included
        return synth.make_field_pocket((40, 37, 42), 0.5, (-10.0, -9.0, -10.5),
                                       lambda x, y, z: 1.0 + 0.3 * np.sin(x) * np.cos(1.3 * y) + 0.2 * np.sin(0.7 * z))
    if name == "flat":       # every inner pose scores the same up to rounding: ties and fallback
        return synth.make_field_pocket((40, 40, 40), 0.5, (-9.75,) * 3,
                                       lambda x, y, z: (np.sqrt(x * x + y * y + z * z) < 9.0) * 1.0)
    if name == "tiny_grid":  # smaller than the ligands: poses leave the padded grid
        return synth.make_field_pocket((5, 4, 6), 0.25, (-0.5, -0.375, -0.625), lambda x, y, z: 1.0 - x * x - y * y)
    if name == "walls":      # a few very large negative voxels beside a shallow field
        v = base.values.copy()
        rng = np.random.Generator(np.random.PCG64(5))
        v[rng.random(v.shape) < 0.002] = -5000.0
        return dataclasses.replace(base, values=v)
    if name == "offset":     # small variation on a large constant
        return synth.make_field_pocket((40, 40, 40), 0.5, (-9.75,) * 3,
                                       lambda x, y, z: 500.0 + np.sin(2.0 * x) + np.cos(1.7 * y + z))
    if name == "negative":
        return dataclasses.replace(base, values=-base.values)
    raise KeyError(name)


@pytest.mark.parametrize("grid", ["f32", "f16"])
@pytest.mark.parametrize("field", ["workload", "faces", "flat", "tiny_grid", "walls", "offset", "negative"])
def test_screening_equals_scoring_every_pose(dk, field, grid):
    pk, db = _field(field), _mixed()
    for align in (1, 5, 6, 9, 30):   # 1, 25, 36, 81 and 900 poses: below, at and past a pass, with and without a tail
        mk = lambda ee: dk.Params.make(restarts=5, align_steps=align, torsion_steps=64, clash_dist=2.0, seed=3,  # noqa: E731
                                       early_exit=ee)
        ref = _run(dk, pk, grid, db, mk(0), (8, -1, 0, 2, 1))
        for shape in ((4, -1, 0, 1, 2), (4, 50, 1, 1, 1), (8, -1, 0, 2, 2), (4, -1, 0, 4, 1), (8, -1, 0, 8, 1)):
            _same(ref, _run(dk, pk, grid, db, mk(1), shape), (field, grid, align, shape))


@pytest.mark.parametrize("align", [32, 127, 128])
def test_screening_at_the_largest_rotation_counts(dk, align):
    """1024, 16129 and 16384 poses: the pass number fills the 9 bits an estimate keeps for it."""
    pk, db = _field("workload"), _mixed(1)
    mk = lambda ee: dk.Params.make(restarts=2, align_steps=align, torsion_steps=8, seed=3, early_exit=ee)  # noqa: E731
    ref = _run(dk, pk, "f32", db, mk(0), (8, -1, 0, 2, 1))
    for shape in ((4, -1, 0, 1, 2), (8, -1, 0, 8, 1)):
        _same(ref, _run(dk, pk, "f32", db, mk(1), shape), (align, shape))


@pytest.mark.parametrize("grid", ["f32", "i16"])
@pytest.mark.parametrize("ligands", [1, 40, 41, 151, 152])
def test_automatic_shapes_change_no_result(dk, ligands, grid):
    """Batch sizes on both sides of the sizes at which a launch changes its shape (8 and 30 ligand-restarts
    per SM: 1,216 and 4,560 on 152 SMs), in every atom bucket."""
    pk = _field("workload")
    if grid == "i16":
        pk = pk.integer(1000)
    db = synth.tile_db(_mixed(1), ligands)
    prm = dk.Params.make(restarts=30, align_steps=8, torsion_steps=32, seed=9)
    _same(_run(dk, pk, grid, db, prm, (4, -1, 0, 4, 1)), _run(dk, pk, grid, db, prm), (ligands, grid))


@pytest.mark.parametrize("clash", [0.0, 0.5, 3.0, 9.0])
def test_bump_check_against_the_oracle(dk, clash):
    """The bump check over four angle passes at once, 100 angles (a last pass partly filled), at thresholds from
    none to most of a molecule: decisions against the oracle, and the same rejected counts whether one or
    eight warps share the check."""
    from oracle import oracle
    from tests import parity
    pk, db = _field("workload"), _mixed(1)
    prm = dk.Params.make(restarts=3, align_steps=8, torsion_steps=100, clash_dist=clash, seed=21)
    res = _run(dk, pk, "f32", db, prm, (4, -1, 0, 1, 1))
    _same(res, _run(dk, pk, "f32", db, prm, (8, -1, 0, 8, 1)), clash)
    op = oracle.Params(restarts=3, align_steps=8, torsion_steps=100, clash_dist=clash, post_align=1, seed=21)
    rep = parity.check(oracle, oracle.GridView.of(pk), db, res, op, threads=8)
    assert not rep.failures, rep.failures[:5]
