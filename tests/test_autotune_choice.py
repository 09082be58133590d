"""The autotuner keeps what it timed (CPU, against a context that only simulates launch times).

With no shape set for a bucket each launch chooses its own, which is not the shape that get_launch reports;
when that choice is the fastest, the context has to be left without a shape set, and a saved table has to
restore it so."""
import time

import numpy as np
import pytest

from paper_2209_05069_gb300 import autotune, synth

REPORTED = dict(warps_per_block=8, smem_carveout_pct=-1, persistent=1, warps_per_item=2, pose_tile=1)


class FakeContext:
    """Launch times by shape: `auto_ms` with no shape set, `ms(shape)` for a set one; a batch takes the slowest
    bucket's time."""

    def __init__(self, auto_ms, ms):
        self.auto_ms, self.ms = auto_ms, ms
        self.shapes = {}

    def set_launch(self, bucket, *shape):
        self.shapes[bucket] = tuple(shape)

    def reset_launch(self, bucket=None):
        for b in (range(5) if bucket is None else [bucket]):
            self.shapes.pop(b, None)

    def get_launch(self, bucket):
        if bucket not in self.shapes:
            return dict(REPORTED)
        return dict(zip(REPORTED, self.shapes[bucket]))

    def batch_create(self, db, params):
        return sorted(set(autotune.bucket_of(np.diff(db.atom_off)).tolist()))

    def batch_launch(self, pocket_id, batch):
        self.cost = max(self.ms(self.shapes[b]) if b in self.shapes else self.auto_ms for b in batch)

    def batch_wait(self, batch):
        t = time.perf_counter() + self.cost * 1e-3
        while time.perf_counter() < t:
            pass

    def batch_destroy(self, batch):
        pass


def _tune(ctx, db):
    return autotune.tune(ctx, 1, db, None, warps=(4, 8), carveouts=(-1,), persistent=(0, 1), warps_per_item=(1, 2),
                         tiles=(1,), reps=1)


@pytest.mark.parametrize("workload", ["uneven", "tiny"])   # several buckets, and one
def test_the_choice_made_by_each_launch_stays_when_it_is_the_fastest(workload):
    db = synth.make_db(synth.WORKLOADS[workload], 24)
    ctx = FakeContext(0.5, lambda shape: 3.0)
    table = _tune(ctx, db)
    assert not ctx.shapes, "a shape was set although the launch's own choice was the fastest"
    table = autotune.confirm(ctx, 1, db, None, table, reps=1)
    assert not ctx.shapes
    assert all(row["automatic"] for row in table.values())
    other = FakeContext(0.5, lambda shape: 3.0)
    autotune.apply(other, table)
    assert not other.shapes


def test_confirm_restores_the_choice_made_by_each_launch():
    db = synth.make_db(synth.WORKLOADS["uneven"], 24)
    ctx = FakeContext(2.0, lambda shape: 0.5)
    table = _tune(ctx, db)
    assert ctx.shapes and not any(row["automatic"] for row in table.values())
    ctx.auto_ms = 0.2   # the whole database favours it
    table = autotune.confirm(ctx, 1, db, None, table, reps=1)
    assert not ctx.shapes and all(row["confirm"]["chosen"] == "library default" for row in table.values())


def test_a_set_shape_stays_when_it_is_the_fastest():
    db = synth.make_db(synth.WORKLOADS["uneven"], 24)
    best = (4, -1, 0, 1, 1)
    ctx = FakeContext(2.0, lambda shape: 0.3 if shape == best else 1.5)
    table = _tune(ctx, db)
    table = autotune.confirm(ctx, 1, db, None, table, reps=1)
    assert set(ctx.shapes.values()) == {best} and set(ctx.shapes) == set(table)
    other = FakeContext(2.0, lambda shape: 1.0)
    autotune.apply(other, table)
    assert other.shapes == ctx.shapes


@pytest.mark.gpu
def test_resolved_shapes_on_a_context():
    from paper_2209_05069_gb300 import dock
    with dock.Context(serve=False) as ctx:
        small, large = ctx.resolve_launch(0, 1), ctx.resolve_launch(0, 10 ** 6)
        assert small["automatic"] and large["automatic"] and small["warps_per_item"] == 8 and large["warps_per_item"] == 1
        ctx.set_launch(0, 4, 60, 1, 2, 1)
        for items in (1, 10 ** 6):
            sh = ctx.resolve_launch(0, items)
            assert not sh.pop("automatic") and sh == ctx.get_launch(0)
        assert ctx.resolve_launch(1, 1)["automatic"]
        ctx.reset_launch(0)
        assert ctx.resolve_launch(0, 1) == small
        with pytest.raises(dock.DockError):
            ctx.resolve_launch(5, 1)
