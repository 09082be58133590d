"""Which serving batches take the latency-oriented shape (8 warps per ligand-restart): dock_config's
serve_latency_items alone decides, with no launch shape set as well.

The counter build shows it: on a trilinear grid an alignment with 8 warps looks every pose up in full, the other
shapes screen the poses by estimates and look up few of them."""
import pytest

from paper_2209_05069_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("option,eight", [(0, True), (-1, False), (100, False), (600, True)])
def test_serve_latency_items_decides(option, eight):
    from paper_2209_05069_gb300 import dock
    w = synth.WORKLOADS["tiny"]
    db = synth.make_db(w, 20)
    prm = dock.Params.make(restarts=30, align_steps=30, torsion_steps=32, seed=5)   # 600 ligand-restarts
    with dock.Context(counters=True, serve_latency_items=option) as ctx:
        pid = ctx.load(synth.workload_pocket(w))
        assert ctx.dock(pid, db, prm) is not None
        work, stats = ctx.exec_counters(), ctx.stats()
    every_pose = 2 * 30 * 900 * int(db.atom_off[-1])
    assert stats["latency_batches"] == (1 if eight else 0)
    assert (work["lookups"] > every_pose) == eight, (work["lookups"], every_pose)
