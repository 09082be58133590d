"""The work a user of this library has it do, as cases that can be timed and compared.

A case is one call (or one small group of calls) through the library's public interface, from a lone
request of a docking service to a screening batch that fills the GPU.  Sizes, pockets and docking
parameters are those of the workloads in ``paper_2209_05069_gb300/synth.py`` (tiny, uneven, large,
serving, plateau) and of the tests' parameter ranges.

Fields of a case:
  mols     the ligands' size distribution: "tiny" (20-30 atoms), "uneven" (10-80), "large" (80-150)
  pocket   the workload whose pocket recipe is used; grid: its storage type, "f32", "f16" or "i16"
  ligands  how many are docked by one pass
  call     "serve": submit / poll / results from host arrays, split over `submissions` tickets;
           "batch": a device-resident batch, launched and its results read back;
           "device": the allocation-free launch, results left in device buffers
  form     of a "batch" call: "batched" or "latency"
  shape    "default", or an explicit launch shape
           "warps per block, carveout, persistent, warps per item, pose tile" for every atom bucket
  restarts, align, torsion, post, early, select_k, best_only   dock_params
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2209_05069_gb300 import dock, synth

# Distinct geometries made for one state; more ligands cycle through them under ids of their own (the
# id keys the starting orientations, so each is docked as new work).
POOL = {"tiny": 96, "uneven": 144, "large": 32}
# Means of the size distributions above: atoms, rotatable bonds, moving atoms per bond.
MEANS = {"tiny": (25.0, 4.0, 3.6), "uneven": (37.9, 5.9, 4.1), "large": (115.0, 30.0, 7.7)}
# Most of the work one pass of a drawn case may have, in pocket lookups: the largest listed case's.
MOST_LOOKUPS = 9.0e9


def _case(name, mols, pocket, grid, ligands, call, **more):
    c = dict(name=name, mols=mols, pocket=pocket, grid=grid, ligands=ligands, call=call, form="batched", shape="default",
             submissions=1, restarts=30, align=30, torsion=256, post=True, early=True, select_k=1, best_only=True)
    c.update(more)
    return c


def listed():
    return [
        # a lone request at a lightly loaded docking service: latency is all that counts
        _case("lone_request", "uneven", "serving", "f32", 1, "serve"),
        # one large molecule docked alone over the whole GPU (the paper's latency design), every output read
        _case("one_large_latency", "large", "large", "f32", 1, "batch", form="latency", best_only=False),
        # the few requests that a service at moderate load has waiting when a stream gets free
        _case("few_requests", "uneven", "serving", "f32", 12, "serve"),
        # a small set of fragments with the parity workload's coarse parameters, all outputs
        _case("fragments", "tiny", "tiny", "f32", 32, "batch", restarts=8, torsion=64, best_only=False),
        # an analogue series: about a hundred ligands against a large FP16 grid
        _case("series", "uneven", "plateau", "f16", 100, "batch"),
        # results kept on the device for a caller's own ranking step, with a coarser and odd angle set,
        # no second alignment and every angle scored in full
        _case("device_ranking", "uneven", "uneven", "f32", 701, "device", align=24, torsion=100, post=False, early=False,
              best_only=False),
        # database screening, the benchmark's size mix, on each kind of grid
        _case("screen_f32", "uneven", "uneven", "f32", 4003, "batch", shape="4,-1,1,1,2"),
        _case("screen_f16", "uneven", "plateau", "f16", 4003, "batch"),
        _case("screen_i16", "uneven", "uneven", "i16", 6007, "batch"),
        # the same screening streamed through the service from host arrays
        _case("screen_served", "uneven", "uneven", "f32", 3000, "serve", submissions=4),
        # large molecules, where the bump check and the scattered gathers weigh most
        _case("large_f32", "large", "large", "f32", 701, "batch"),
        # large molecules on an FP16 grid with several poses kept per ligand, all outputs
        _case("large_f16_poses", "large", "large", "f16", 501, "batch", select_k=4, best_only=False),
    ]


def draw(rng):
    mols = rng.choice(["tiny", "uneven", "uneven", "uneven", "large"])
    pocket = {"tiny": ["tiny", "uneven"], "uneven": ["uneven", "serving", "plateau"], "large": ["large", "plateau"]}[mols]
    c = _case("", mols, rng.choice(pocket), rng.choice(["f32", "f32", "f16", "i16"]), 1,
              rng.choice(["batch", "batch", "serve", "device"]))
    del c["name"]
    c["restarts"] = rng.choice([30, 30, rng.randint(4, 40)])
    c["align"] = rng.choice([30, 30, rng.randint(10, 36)])
    c["torsion"] = rng.choice([256, 256, rng.randint(60, 360)])
    c["post"] = rng.random() < 0.85
    c["early"] = rng.random() < 0.85
    c["best_only"] = rng.random() < 0.6
    most = MOST_LOOKUPS / _lookups_per_ligand(c)
    if c["call"] == "device":  # the fixed scratch of the allocation-free launch
        most = min(most, 0.8 * dock.NOALLOC_SCRATCH_BYTES / (12 * MEANS[mols][0] * 1.15 * c["restarts"]))
    c["ligands"] = max(1, int(math.exp(rng.uniform(0.0, math.log(max(2.0, min(most, 6000.0)))))))
    if c["call"] == "serve":
        c["submissions"] = rng.randint(1, min(4, c["ligands"]))
    if c["call"] == "batch":
        if c["ligands"] <= 24 and rng.random() < 0.5:
            c["form"] = "latency"
        elif rng.random() < 0.3:
            c["shape"] = rng.choice(["4,-1,1,1,2", "8,-1,1,2,2", "8,-1,1,2,1", "8,-1,0,8,1", "8,-1,0,1,1", "4,60,0,4,1"])
        if rng.random() < 0.25:
            c["select_k"] = rng.randint(2, 4)
    return c


def _lookups_per_ligand(c):
    """Pocket lookups the method makes for one ligand of mean size (every angle scored)."""
    n, b, m = MEANS[c["mols"]]
    return c["restarts"] * ((1 + bool(c["post"])) * c["align"] ** 2 * n + b * c["torsion"] * m + n)


# ---- what a program has in hand ----------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _context(shape):
    """One context per launch shape, kept by the program for as long as it runs."""
    ctx = dock.Context()
    if shape != "default":
        for bucket in range(5):
            ctx.set_launch(bucket, *[int(v) for v in shape.split(",")])
    return ctx


def _pocket(case, seed):
    w = synth.WORKLOADS[case["pocket"]]
    pk = synth.make_pocket(w.grid, w.spacing, w.radius, w.noise, synth.pocket_seed(w) + 7919 * seed)
    return pk.integer() if case["grid"] == "i16" else pk


@functools.lru_cache(maxsize=None)
def _reference_pool(mols):
    """The workload's own first ligands: their sizes are those of every state, whatever its seed."""
    return synth.make_db(synth.WORKLOADS[mols], POOL[mols])


def _ligands(case, seed):
    """`ligands` ligands of the seed's own geometries: each is grown anew with the atom and rotatable-bond counts of the
    workload's ligand of its number (redrawn where a grown tree has too few rotatable bonds)."""
    n, ref = case["ligands"], _reference_pool(case["mols"])
    pool = []
    for l in range(min(n, ref.n_lig)):
        rng = np.random.Generator(np.random.PCG64([synth.BASE_SEED, 104729 + seed, l]))
        for _ in range(200):
            xyz, bonds, rot, clipped = synth.make_ligand(rng, ref.n_atoms(l), ref.n_rot(l))
            if not clipped:
                break
        else:
            xyz, bonds, rot, _ = ref.ligand(l)
        pool.append((xyz, bonds, rot, l))
    return synth.tile_db(synth.from_ligands(pool), n, first_id=1000003 * (seed % 1009))


def _params(case):
    return dock.Params.make(restarts=case["restarts"], align_steps=case["align"], torsion_steps=case["torsion"],
                            clash_dist=2.0, post_align=int(case["post"]), early_exit=int(case["early"]), seed=20905069,
                            select_k=case["select_k"],
                            outputs=dock.DOCK_OUTPUT_BEST if case["best_only"] else dock.DOCK_OUTPUT_FULL)


class _State:
    def __init__(self, case, seed):
        self.case = case
        self.ctx = _context(case["shape"])
        self.params = _params(case)
        self.pocket = self.ctx.load(_pocket(case, seed), case["grid"])
        db = _ligands(case, seed)
        self.batch = None
        if case["call"] == "serve":
            edges = np.linspace(0, db.n_lig, case["submissions"] + 1).astype(int)
            self.parts = [db.slice(int(a), int(b)) for a, b in zip(edges[:-1], edges[1:])]
            return
        self.batch = self.ctx.batch_create(db, self.params)
        if case["call"] == "device":
            R, L, A, B = self.params.restarts, db.n_lig, int(db.atom_off[-1]), int(db.rot_off[-1])
            f = lambda *s: torch.zeros(*s, device="cuda")  # noqa: E731
            i = lambda *s: torch.zeros(*s, device="cuda", dtype=torch.int32)  # noqa: E731
            self.out = dict(score=f(L), best_restart=i(L), xyz=f(A, 3), clash_count=i(L), restart_score=f(L * R),
                            restart_clash=i(L * R), align_idx=i(L * R), post_idx=i(L * R), torsion_idx=i(max(1, B * R)),
                            rejected=i(max(1, B * R)))

    def __del__(self):
        try:
            if self.batch is not None:
                self.ctx.batch_destroy(self.batch)
            self.ctx.unload_pocket(self.pocket)
        except Exception:  # the interpreter is going down
            pass


def prepare(case, seed):
    return _State(case, seed)


def _values(r):
    """A pass's results without the service's clock readings."""
    return {k: v for k, v in r.items() if k != "latency_ns"}


def run(state):
    ctx, case = state.ctx, state.case
    if case["call"] == "serve":
        tickets = [ctx.submit(state.pocket, part, state.params) for part in state.parts]
        out = []
        for t in tickets:
            ctx.poll(t, -1)
            out.append(_values(ctx.results(t)))
        return out
    if case["call"] == "device":
        ctx.batch_launch_noalloc(state.pocket, state.batch, {k: v.data_ptr() for k, v in state.out.items()},
                                 torch.cuda.current_stream().cuda_stream)
        return state.out
    form = dock.DOCK_FORM_LATENCY if case["form"] == "latency" else dock.DOCK_FORM_BATCHED
    ctx.batch_launch(state.pocket, state.batch, form)
    return _values(ctx.batch_results(state.batch))


def work(case):
    """Each ligand and the pocket's voxels read once, each result written once; per lookup 8 multiply-adds to
    place the atom and, on a trilinear grid, 7 differences and 7 multiply-adds to interpolate."""
    n, b, _ = MEANS[case["mols"]]
    L, R = case["ligands"], case["restarts"]
    voxel = {"f32": 4, "f16": 2, "i16": 2}[case["grid"]]
    w = synth.WORKLOADS[case["pocket"]]
    out = 12 + 12 * n * max(1, case["select_k"]) + (0 if case["best_only"] else 16 * R + 8 * R * b)
    flops = 17 if case["grid"] == "i16" else 38
    return {"bytes": L * (12 * n + 8 * n + 8 * b + out) + voxel * w.grid ** 3, "flops": flops * L * _lookups_per_ligand(case)}


# ---- the same in 64 bits -----------------------------------------------------------------------------

def _grid_lookup(case, pk):
    """The pocket's value at positions (..., 3), in 64 bits."""
    v = torch.as_tensor(pk.values, device="cuda")
    v = (v.half() if case["grid"] == "f16" else v).double()
    o = torch.tensor([float(np.float32(x)) for x in pk.origin], device="cuda", dtype=torch.float64)
    h = float(np.float32(pk.spacing))
    n = torch.tensor(pk.dims, device="cuda")
    flat = v.reshape(-1)
    nx, ny, _ = pk.dims

    def nearest(x):
        i = torch.floor((x - o) / h + 0.5).long()
        ok = ((i >= 0) & (i < n)).all(-1)
        i = torch.minimum(i.clamp(min=0), n - 1)
        return torch.where(ok, flat[(i[..., 2] * ny + i[..., 1]) * nx + i[..., 0]], 0.0)

    def trilinear(x):
        u = (x - o) / h
        ok = ((u >= 0) & (u <= n - 1)).all(-1)
        i = torch.minimum(torch.floor(u).long().clamp(min=0), n - 2)
        t = u - i
        at = (i[..., 2] * ny + i[..., 1]) * nx + i[..., 0]
        s = torch.zeros_like(at, dtype=torch.float64)
        for dz in (0, 1):
            for dy in (0, 1):
                for dx in (0, 1):
                    wt = ((t[..., 0] if dx else 1 - t[..., 0]) * (t[..., 1] if dy else 1 - t[..., 1]) *
                          (t[..., 2] if dz else 1 - t[..., 2]))
                    s += wt * flat[at + (dz * ny + dy) * nx + dx]
        return torch.where(ok, s, 0.0)

    return nearest if case["grid"] == "i16" else trilinear


def _starts(case, lig_id, seed):
    """Rotation matrices of the starting orientations: the identity, then Shoemake's uniform rotations from
    SplitMix64 draws keyed by the ligand's id."""
    mask = (1 << 64) - 1

    def mix(state, k):
        z = (state + k * 0x9E3779B97F4A7C15) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        return z ^ (z >> 31)

    key = mix(seed ^ lig_id, 1)
    out = [np.eye(3)]
    for r in range(1, case["restarts"]):
        u = [(mix(key, 3 * r + t + 1) >> 40) / 2.0 ** 24 for t in range(3)]
        a, b = math.sqrt(1 - u[0]), math.sqrt(u[0])
        x, y = a * math.sin(2 * math.pi * u[1]), a * math.cos(2 * math.pi * u[1])
        z, w = b * math.sin(2 * math.pi * u[2]), b * math.cos(2 * math.pi * u[2])
        out.append(np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                             [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                             [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]]))
    return torch.as_tensor(np.stack(out), device="cuda")


def _moving_side(n, bonds, a, b):
    near = [[] for _ in range(n)]
    for p, q in bonds:
        near[p].append(int(q))
        near[q].append(int(p))
    seen, todo = {b}, [b]
    while todo:
        v = todo.pop()
        for q in near[v]:
            if q not in seen and not (v == b and q == a):
                seen.add(q)
                todo.append(q)
    return sorted(seen)


def _dock64(case, value, centre, xyz, bonds, rot, lig_id, seed):
    """Every restart's final score of one ligand, in 64 bits."""
    n, R, N, A = len(xyz), case["restarts"], case["align"], case["torsion"]
    f64 = dict(device="cuda", dtype=torch.float64)
    x = torch.as_tensor(np.asarray(xyz, np.float64), device="cuda")
    pose = centre + torch.einsum("rij,aj->rai", _starts(case, lig_id, seed), x - x.mean(0))
    ang = 2 * math.pi * torch.arange(N, **f64) / N
    c, s, o, one = ang.cos(), ang.sin(), torch.zeros(N, **f64), torch.ones(N, **f64)
    rx = torch.stack([one, o, o, o, c, -s, o, s, c], -1).reshape(N, 3, 3)
    ry = torch.stack([c, o, s, o, one, o, -s, o, c], -1).reshape(N, 3, 3)
    turns = torch.einsum("jab,ibc->ijac", ry, rx).reshape(N * N, 3, 3)

    def align(pose):
        mid = pose.mean(1, keepdim=True)
        rel = pose - mid
        score = torch.stack([value(mid[r] + torch.einsum("fij,aj->fai", turns, rel[r])).sum(-1).argmax() for r in range(R)])
        return mid + torch.einsum("rij,raj->rai", turns[score], rel)

    pose = align(pose)
    th = 2 * math.pi * torch.arange(A, **f64) / A
    ct, st = th.cos()[None, :, None, None], th.sin()[None, :, None, None]
    for a, b in rot:
        a, b = int(a), int(b)
        mv = [i for i in _moving_side(n, bonds, a, b) if i != b]
        fx = [i for i in range(n) if i not in mv and i not in (a, b)]
        axis = pose[:, b] - pose[:, a]
        axis = (axis / axis.norm(dim=-1, keepdim=True))[:, None, None]
        v = (pose[:, mv] - pose[:, b:b + 1])[:, None]
        along = (v * axis).sum(-1, keepdim=True) * axis
        r = v - along
        at = pose[:, b][:, None, None] + along + ct * r + st * torch.linalg.cross(axis.expand_as(r), r, dim=-1)  # (R, A, m, 3)
        bump = torch.zeros(R, A, dtype=torch.bool, device="cuda")
        for j in fx:
            if mv:
                bump |= (((at - pose[:, j][:, None, None]) ** 2).sum(-1) < 4.0).any(-1)
        score = value(at).sum(-1).masked_fill(bump, -math.inf)
        k = torch.where(bump.all(-1), torch.zeros(R, dtype=torch.long, device="cuda"), score.argmax(-1))
        if mv:
            pose = pose.clone()
            pose[:, mv] = at[torch.arange(R, device="cuda"), k]
    if case["post"]:
        pose = align(pose)
    return value(pose).sum(-1)


def exact(case, seed):
    """The scores in 64 bits, for the cases small enough.  Indices are whole numbers, and a pose has no value of its
    own here: a choice between two poses whose scores agree to the last bits of 32 leads to either."""
    if case["ligands"] * _lookups_per_ligand(case) > 1.5e8:
        return None
    pk = _pocket(case, seed)
    h = float(np.float32(pk.spacing))
    value = _grid_lookup(case, pk)
    centre = torch.tensor([float(np.float32(o)) + h * (n - 1) / 2 for o, n in zip(pk.origin, pk.dims)], device="cuda",
                          dtype=torch.float64)
    db = _ligands(case, seed)
    scores = []
    for l in range(db.n_lig):
        xyz, bonds, rot, lig_id = db.ligand(l)
        scores.append(_dock64(case, value, centre, xyz, bonds, rot, lig_id, 20905069))
    scores = torch.stack(scores)  # (ligands, restarts)

    def outputs(a, b):
        s = scores[a:b]
        o = dict(score=s.max(1).values, best_restart=None, xyz=None, clash_count=None)
        if not case["best_only"] or case["call"] == "device":
            o.update(restart_score=s.reshape(-1), restart_clash=None, align_idx=None, post_idx=None, torsion_idx=None,
                     rejected=None)
        if case["call"] != "device":
            o.update(select_restart=None, select_score=s.max(1).values if case["select_k"] == 1 else None, select_xyz=None)
        return o

    if case["call"] != "serve":
        return outputs(0, db.n_lig)
    edges = np.linspace(0, db.n_lig, case["submissions"] + 1).astype(int)
    return [outputs(int(a), int(b)) for a, b in zip(edges[:-1], edges[1:])]
