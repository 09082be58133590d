"""Screening cells at the limits of their layout: an axis of 1,968 voxels (the longest that the fixed-point coordinates
hold) and one beyond it, and a grid whose rows are lengthened so that the biased cell index stays below 2^32.

Every output equals that of scoring each pose in full, bit for bit, and the counter build tells whether the poses were
screened (loads that are not lookups)."""
import numpy as np
import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu


def _rows_lengthened(nx, ny, nz):
    """Whether bias + cells of the unlengthened layout reach 2^32 (32 cells of padding per axis)."""
    cx, cy, cz = nx + 31, ny + 31, nz + 31
    return (0x45000 * (cy * cx + cx + 1)) % 2 ** 32 + cx * cy * cz >= 2 ** 32


@pytest.mark.parametrize("grid", ["f32", "f16"])
@pytest.mark.parametrize("dims,lengthened,screened", [((67, 123, 77), True, True), ((124, 66, 78), True, True),
                                                      ((1968, 24, 24), False, True), ((24, 1968, 24), False, True),
                                                      ((24, 24, 1968), False, True), ((1969, 24, 24), False, False)])
def test_layout_limits(dims, lengthened, screened, grid):
    from paper_2209_05069_gb300 import dock
    assert _rows_lengthened(*dims) == lengthened
    h = 0.75
    rng = np.random.Generator(np.random.PCG64(4))
    v = rng.random(dims[::-1]).astype(np.float32)
    for axis in range(3):   # zero faces
        np.moveaxis(v, axis, 0)[[0, -1]] = 0
    origin = [-h * (n - 1) / 2 for n in dims]
    db = synth.make_db(synth.WORKLOADS["tiny"], 12)
    got = {}
    for early in (0, 1):
        prm = dock.Params.make(restarts=6, align_steps=30, torsion_steps=32, seed=5, early_exit=early)
        with dock.Context(serve=False, counters=True) as ctx:
            for b in range(5):
                ctx.set_launch(b, 4, -1, 0, 1, 2)
            batch = ctx.batch_create(db, prm)
            ctx.batch_launch(ctx.load_pocket(v, h, origin, grid), batch)
            got[early] = ctx.batch_results(batch), ctx.exec_counters()
            ctx.batch_destroy(batch)
    for k in got[0][0]:
        assert np.array_equal(got[0][0][k], got[1][0][k]), k
    # the memory bound of one pocket: the cells of a thin grid on FP16, half the size of FP32's, are too small beside them
    own = (32 if grid == "f32" else 16) * int(np.prod([n - 1 for n in dims]))
    fits = 8 * int(np.prod([n + 31 for n in dims])) <= max(16 << 20, 2 * own)
    assert (got[1][1]["loads"] > got[1][1]["lookups"]) == (screened and fits)
    assert fits or grid == "f16"
