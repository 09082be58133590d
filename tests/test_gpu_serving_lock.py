"""Calls on a context are not held up while its serving loop watches a young batch.

The loop looks at a small running batch without sleeping.  It does so without the context's lock: a call that needs
the lock meanwhile (here dock_poll without waiting, from one thread) takes as long as on an idle context, up to the
short times in which the loop packs a batch or hands results over (1 call in 20 is allowed for them)."""
import time

import numpy as np
import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu


def test_poll_is_not_held_up_by_the_watch():
    from paper_2209_05069_gb300 import dock
    db = synth.make_db(synth.WORKLOADS["uneven"], 12)
    prm = dock.Params.make(restarts=30, seed=5, outputs=dock.DOCK_OUTPUT_BEST)   # 360 ligand-restarts: a small batch

    def poll_us(ctx, ticket):
        t = time.perf_counter()
        rc, _ = ctx.poll(ticket, 0)
        return (time.perf_counter() - t) * 1e6, rc

    with dock.Context() as ctx:
        pid = ctx.load(synth.workload_pocket(synth.WORKLOADS["serving"]))
        for _ in range(5):
            ctx.dock(pid, db, prm)
        done = ctx.submit(pid, db, prm)
        ctx.poll(done, -1)
        time.sleep(0.01)
        idle = [poll_us(ctx, done)[0] for _ in range(2000)]
        ctx.results(done)
        busy = []
        for _ in range(100):
            ticket = ctx.submit(pid, db, prm)
            rc = dock.DOCK_PENDING
            while rc == dock.DOCK_PENDING:
                us, rc = poll_us(ctx, ticket)
                busy.append(us)
            ctx.results(ticket)
    p_idle, p_busy = np.percentile(idle, 95), np.percentile(busy, 95)
    print(f"\npoll, 95th percentile: idle {p_idle:.2f} us, beside a watched batch {p_busy:.2f} us ({len(busy)} calls)")
    assert p_busy < 2.0 * p_idle + 2.0
