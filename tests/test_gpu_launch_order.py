"""Launch order and the driver's carveout: on the integer grid with one warp per item and a pose tile of 1 the buckets of
a full batch share the GPU without starving one another of L1.

An SM keeps the carveout of the first kernel it runs.  With the largest molecules first, whose 32 items per SM take
211 KB, the batch below ran 2.7 times as long as with a carveout set; with the bulk of the work first 1.3 times.
The line lies between, and the fastest of several runs counts."""
import time

import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("persistent", [0, 1])
def test_integer_grid_keeps_its_l1(persistent):
    from paper_2209_05069_gb300 import dock
    w = synth.WORKLOADS["uneven"]
    db = synth.tile_db(synth.make_db(w, 400), 4000)
    prm = dock.Params.make(restarts=30, align_steps=30, torsion_steps=256, seed=7)
    best = {}
    with dock.Context(serve=False) as ctx:
        pid = ctx.load(synth.workload_pocket(w).integer(1000), "i16")
        batch = ctx.batch_create(db, prm)
        for carveout in (-1, 60):
            for b in range(5):
                ctx.set_launch(b, 8, carveout, persistent, 1, 1)
            times = []
            for _ in range(8):
                t = time.perf_counter()
                ctx.batch_launch(pid, batch)
                ctx.batch_wait(batch)
                times.append(time.perf_counter() - t)
            best[carveout] = min(times)
        ctx.batch_destroy(batch)
    print(f"\npersistent {persistent}: driver's carveout {best[-1] * 1e3:.2f} ms, 60% {best[60] * 1e3:.2f} ms")
    assert best[-1] < 1.9 * best[60]
