"""Device memory of a loaded pocket: its cells, and screening cells only where they are used and within their bounds."""
import numpy as np
import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _taken(load):
    """Device bytes taken by load() and kept after it."""
    torch = pytest.importorskip("torch")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    load()
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0]


def _estimates(pk, grid):
    from paper_2209_05069_gb300 import dock
    with dock.Context(serve=False, counters=True) as ctx:
        for b in range(5):
            ctx.set_launch(b, 4, -1, 0, 1, 2)
        db = synth.make_db(synth.WORKLOADS["tiny"], 4)
        batch = ctx.batch_create(db, dock.Params.make(restarts=4, torsion_steps=8, seed=3))
        ctx.batch_launch(ctx.load(pk, grid), batch)
        ctx.batch_wait(batch)
        work = ctx.exec_counters()
        ctx.batch_destroy(batch)
    return work["loads"] > work["lookups"]


def test_a_refused_field_takes_no_screening_memory():
    """160^3 voxels: 64 MiB of FP16 cells, 53 MiB of screening cells.  The pool takes memory in blocks of 32 MiB."""
    from paper_2209_05069_gb300 import dock
    mk = lambda f: synth.make_field_pocket((160,) * 3, 0.375, (-29.8,) * 3, f)  # noqa: E731
    used = mk(lambda x, y, z: np.sin(x) * np.cos(y + z))
    refused = mk(lambda x, y, z: 5000.0 + np.sin(x) * np.cos(y + z))
    for pk, lo, hi in ((used, 110 * MB, 160 * MB), (refused, 60 * MB, 100 * MB)):
        with dock.Context(serve=False) as ctx:
            warm = ctx.load(synth.workload_pocket(synth.WORKLOADS["tiny"]))
            assert lo <= _taken(lambda: ctx.load(pk, "f16")) <= hi
            ctx.unload_pocket(warm)


@pytest.mark.parametrize("dims", [(2, 2, 1900), (1900, 2, 3), (40, 1900, 3)])
def test_a_thin_grid_takes_none_beyond_its_bound(dims):
    from paper_2209_05069_gb300 import dock
    rng = np.random.Generator(np.random.PCG64(3))
    values = rng.random(dims[::-1]).astype(np.float32)
    with dock.Context(serve=False) as ctx:
        taken = _taken(lambda: [ctx.load_pocket(values, 0.375, (0, 0, 0)) for _ in range(8)])
    own = 8 * 32 * int(np.prod([d - 1 for d in dims]))
    assert taken <= 3 * own + 8 * 16 * MB + 64 * MB   # without the bound: 8 x 17 to 73 MB more


def test_screening_cells_of_all_pockets_are_bounded():
    """Thin grids whose screening cells take just under the 16 MiB of one pocket's bound: 1/16 of the device's memory is
    reached after about a thousand, later pockets load without, and unloading makes room again."""
    torch = pytest.importorskip("torch")
    from paper_2209_05069_gb300 import dock
    total = torch.cuda.mem_get_info()[1]
    nz = 1770                                            # 33 x 33 x 1,801 cells of 8 bytes: 14.96 MiB
    each = 8 * 33 * 33 * (nz - 1 + 32)
    count = total // 16 // each + 200
    values = np.random.Generator(np.random.PCG64(3)).random((nz, 2, 2)).astype(np.float32)
    with dock.Context(serve=False) as ctx:
        pids = []
        taken = _taken(lambda: pids.extend(ctx.load_pocket(values, 0.375, (0, 0, 0)) for _ in range(count)))
        assert 0.9 * total / 16 <= taken <= total / 16 + 512 * MB
        for p in pids:
            ctx.unload_pocket(p)
        one = synth.workload_pocket(synth.WORKLOADS["tiny"])
        assert _taken(lambda: [ctx.load_pocket(values, 0.375, (0, 0, 0)) for _ in range(20)]) <= 1024 * MB
    assert _estimates(one, "f32")
