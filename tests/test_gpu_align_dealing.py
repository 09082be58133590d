"""An alignment that is not screened deals its poses to an item's warps by single passes of 32.

Times, on one batch: with 4 warps per item 64 poses (8 angles per axis) take as long as 25 (5 angles), for either
way each warp has at most one pass; dealt in blocks of 64 one warp has two, which took 1.29 times as long.  Between
them 1.15, and the fastest of several runs."""
import time

import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", ["f32", "f16"])
def test_two_passes_on_two_warps(grid):
    from paper_2209_05069_gb300 import dock
    w = synth.WORKLOADS["uneven"]
    db = synth.tile_db(synth.make_db(w, 200), 1000)
    best = {}
    with dock.Context(serve=False) as ctx:
        for b in range(5):
            ctx.set_launch(b, 8, -1, 1, 4, 1)
        pid = ctx.load(synth.workload_pocket(w), grid)
        for n in (5, 8):
            prm = dock.Params.make(restarts=30, align_steps=n, torsion_steps=64, seed=7, early_exit=0)
            batch = ctx.batch_create(db, prm)
            times = []
            for _ in range(12):
                t = time.perf_counter()
                ctx.batch_launch(pid, batch)
                ctx.batch_wait(batch)
                times.append(time.perf_counter() - t)
            ctx.batch_destroy(batch)
            best[n] = min(times)
    print(f"\n{grid}: 25 poses {best[5] * 1e3:.3f} ms, 64 poses {best[8] * 1e3:.3f} ms")
    assert best[8] < 1.15 * best[5]
