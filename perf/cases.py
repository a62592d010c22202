"""Timed cases: what a program that uses the mesher has it do, through the package's
public calls, over the sizes and kinds of input that the repository's own
configurations (``meshgen.CONFIGS``, the batch and served workloads) and tests use.

A case names an operation and its input:

* ``run``     ``Mesh.run`` on a triangulation resident on the GPU (Algorithm 1 whole),
              then its polygons: the main path, from a thousand points to ten million.
* ``phases``  the same method one phase at a time (label, seeds, traversal,
              reparation), with the polygons of both passes, the seeds and the
              longest-edge paths: a program that looks at the intermediate results.
* ``batch``   many small and medium meshes as one batch, with its tuned schedule.
* ``serve``   a burst of requests from pinned host buffers to the native server.
* ``host``    one mesh from pinned host buffers and its polygons back to the host, the
              twin array built on the device from the triangles alone.
* ``twin``    the twin and Trivertex arrays of a triangulation that comes without them.
"""
from __future__ import annotations

import functools

import numpy as np
import torch

import meshgen
import paper_2204_05438_gb300 as pg

# Meshes up to this many points are triangulated anew for each seed; a larger one
# (a second of host time per million points) is triangulated once per process, and
# each seed meshes another quarter turn and shear of it.
FRESH_POINTS = 2_000_000


def listed() -> list[dict]:
    return [
        # the smallest calls: one launch, latency and host work count
        {"name": "run-uniform-1k", "op": "run", "kind": "uniform", "n": 1_000},
        {"name": "run-gmm-1500", "op": "run", "kind": "gmm", "n": 1_500},
        # a part with a notch and holes (borders, tips at the borders), tens of
        # thousands of triangles: the launches and the longest chains count
        {"name": "run-holes-20k", "op": "run", "kind": "holes", "n": 20_011},
        # an ordinary graded mesh
        {"name": "run-gmm-200k", "op": "run", "kind": "gmm", "n": 200_003},
        # a uniform mesh of the paper's smallest size
        {"name": "run-uniform-1m", "op": "run", "kind": "uniform", "n": 1_000_000},
        # triangles in no order, as a refining triangulator may leave them
        {"name": "run-shuffled-1m", "op": "run", "kind": "shuffled", "n": 1_000_000},
        # the largest: the benchmark's workload
        {"name": "run-gmm-10m", "op": "run", "kind": "gmm", "n": 10_000_000},
        # the method phase by phase
        {"name": "phases-gmm-700k", "op": "phases", "kind": "gmm", "n": 700_001},
        # a batch of meshes, sizes as in the batch workload
        {"name": "batch-400", "op": "batch", "kind": "mixed", "n": 50_000, "count": 400},
        # requests from the host, sizes as in the served workload
        {"name": "serve-24", "op": "serve", "kind": "mixed", "n": 200_000, "count": 24},
        # one mesh from the host without its twin array
        {"name": "host-uniform-500k", "op": "host", "kind": "uniform", "n": 500_000},
        # the triangulation's topology alone
        {"name": "twin-gmm-2m", "op": "twin", "kind": "gmm", "n": 2_000_000},
    ]


def _size(rng, lo: int, hi: int) -> int:
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng) -> dict:
    op = rng.choice(["run", "run", "run", "run", "phases", "batch", "serve", "host", "twin"])
    if op == "batch":
        return {"op": op, "kind": "mixed", "n": _size(rng, 2_000, 100_000),
                "count": _size(rng, 16, 600)}
    if op == "serve":
        return {"op": op, "kind": "mixed", "n": _size(rng, 2_000, 400_000),
                "count": rng.randint(3, 30)}
    kinds = ["uniform", "gmm", "shuffled"] + (["holes"] if op in ("run", "phases") else [])
    kind = rng.choice(kinds)
    # a carved domain is cut on the host in numpy: smaller, to keep that short
    hi = 400_000 if kind == "holes" else (5_000_000 if op == "run" else 2_000_000)
    return {"op": op, "kind": kind, "n": _size(rng, 300, hi)}


# ------------------------------------------------------------------ inputs
def _side(n: int) -> int:
    """The lattice: 2^20 for small meshes, 2^24 and 2^26 for larger ones, as in the
    named configurations."""
    return 1 << (20 if n <= 20_000 else (24 if n <= 2_000_000 else 26))


@functools.lru_cache(maxsize=1)
def _large(kind: str, n: int) -> dict:
    for name, cfg in meshgen.CONFIGS.items():
        if (cfg["kind"], cfg["n"], cfg["side"]) == (kind, n, _side(n)):
            return meshgen.load(name)
    return meshgen.generate(kind, n, _side(n), 2)


def _turned(mesh: dict, side: int, seed: int) -> dict:
    """The same triangles after a quarter turn and a shear, exact on the lattice
    (coordinates stay below 16 * side <= 2^30, every triangle keeps its orientation)."""
    x, y = mesh["xy"][:, 0], mesh["xy"][:, 1]
    for _ in range((seed // 16) % 4):
        x, y = side - 1 - y, x
    xy = np.stack([13 * x + (seed % 4) * y, 13 * y + (seed // 4 % 4) * x], axis=1)
    return {"xy": xy, "tri": mesh["tri"], "twin": mesh["twin"]}


def _mesh(kind: str, n: int, seed: int) -> dict:
    if kind == "holes":
        return meshgen.domain_with_holes("uniform", n, _side(n), seed)
    base = "uniform" if kind == "shuffled" else kind
    if n <= FRESH_POINTS:
        mesh = meshgen.generate(base, n, _side(n), seed)
    else:
        mesh = _turned(_large(base, n), _side(n), seed)
    return meshgen.shuffled(mesh, seed) if kind == "shuffled" else mesh


def _plan(case: dict, nmin: int) -> dict:
    """Point counts log-uniform in [nmin, n] and kinds, the same for every seed."""
    return meshgen.batch_plan(case["count"], 11, nmin=nmin, nmax=case["n"])


def _meshes(plan: dict, seed: int) -> list[dict]:
    seeds = np.random.default_rng(seed).integers(1, 2**62, len(plan["ns"])).astype(np.uint64)
    return meshgen.batch(plan["ns"], seeds, plan["kinds"], plan["sides"])


def _pinned(a, dtype) -> torch.Tensor:
    return torch.as_tensor(np.ascontiguousarray(a)).to(dtype).pin_memory()


def _csr(n: int, **kw) -> tuple[torch.Tensor, torch.Tensor]:
    """Offsets and vertices of any polygon mesh over n points (at most 2n triangles)."""
    return torch.zeros(2 * n + 1, dtype=torch.int64, **kw), torch.zeros(6 * n, dtype=torch.int32, **kw)


class _Kept:
    """The program's own copies of results: a handle lends its buffers only until its
    next call.  Sized for any mesh of n points; each pass fills the front."""

    def __init__(self, n: int, names: str):
        off, vtx = _csr(n, device="cuda")
        tri = torch.zeros(2 * n, dtype=torch.int32, device="cuda")
        like = {"off": off, "vtx": vtx, "labels": tri.to(torch.uint8)}
        self.to = {k: like.get(k.rstrip("0"), tri).clone() for k in names.split()}

    def keep(self, **got) -> dict:
        for k, t in got.items():
            self.to[k][:t.numel()].copy_(t)
        return {**self.to, **{"n_" + k: t.numel() for k, t in got.items()}}


class _Handle:
    """A handle that owns its device inputs, destroyed with its state."""

    def __init__(self, n: int, m: int):
        self.handle = pg.mesh_create_host(n, m)

    def __del__(self):
        pg.mesh_destroy(self.handle)


class _Requests:
    """A server with its requests' pinned buffers, its slots made by a first burst."""

    def __init__(self, meshes: list[dict]):
        self.server = pg.Server(16 << 30, max_slots=16)
        self.args = []
        for mesh in meshes:
            self.args.append((_pinned(mesh["xy"], torch.int64), _pinned(mesh["tri"], torch.int32),
                              _pinned(mesh["twin"], torch.int32),
                              *_csr(mesh["xy"].shape[0], pin_memory=True)))
        self.burst()

    def burst(self) -> list:
        ids = [self.server.submit(*a) for a in self.args]
        left = set(ids)
        while left:
            for r in self.server.poll(wait_us=1000):
                if r["status"] != 0:
                    raise RuntimeError(pg.status_str(r["status"]))
                left.discard(r["id"])
        return [a[3:] for a in self.args]


def prepare(case: dict, seed: int) -> dict:
    op = case["op"]
    if op == "batch":
        plan = _plan(case, 200)
        batch = pg.batch_from_numpy(meshgen.concat(_meshes(plan, seed)))
        batch.tune()
        return {"op": op, "batch": batch, "out": _Kept(int(plan["ns"].sum()), "off vtx"),
                "first": torch.zeros(case["count"] + 1, dtype=torch.int64, device="cuda")}
    if op == "serve":
        return {"op": op, "requests": _Requests(_meshes(_plan(case, 1_000), seed))}
    mesh = _mesh(case["kind"], case["n"], seed)
    if op == "run":
        return {"op": op, "mesh": pg.from_numpy(mesh), "out": _Kept(case["n"], "off vtx")}
    if op == "phases":
        return {"op": op, "mesh": pg.from_numpy(mesh),
                "out": _Kept(case["n"], "seeds off0 vtx0 region depth off vtx labels")}
    n, m = mesh["xy"].shape[0], mesh["tri"].shape[0]
    if op == "host":
        return {"op": op, "own": _Handle(n, m), "xy": _pinned(mesh["xy"], torch.int64),
                "tri": _pinned(mesh["tri"], torch.int32), "csr": _csr(n, pin_memory=True)}
    # a handle sized for any triangulation of n points, then for this one
    own = _Handle(n, 2 * n)
    xy, tri, twin = pg.mesh_inputs(own.handle, n, 2 * n)
    xy.copy_(torch.as_tensor(mesh["xy"].reshape(-1)))
    tri[:3 * m].copy_(torch.as_tensor(mesh["tri"].reshape(-1)))
    twin.zero_()
    twin.own = own  # a view of the handle's buffer
    torch.cuda.synchronize()
    pg.mesh_set_size(own.handle, n, m)
    return {"op": op, "own": own, "n": n, "twin": twin}


# ------------------------------------------------------------------ one pass
def run(state: dict):
    op = state["op"]
    if op == "run":
        state["mesh"].run()
        off, vtx = state["mesh"].polygons()
        return state["out"].keep(off=off, vtx=vtx)
    if op == "phases":
        mesh, out = state["mesh"], state["out"]
        mesh.label()
        mesh.seeds()
        mesh.traverse()
        off0, vtx0 = mesh.polygons()
        region, depth = mesh.lepp()
        out.keep(off0=off0, vtx0=vtx0, region=region, depth=depth)
        mesh.repair()
        off, vtx = mesh.polygons()
        return out.keep(seeds=mesh.seed_list(), off=off, vtx=vtx, labels=mesh.labels())
    if op == "batch":
        state["batch"].run()
        off, vtx, first = state["batch"].all_polygons()
        state["first"].copy_(first)
        return {**state["out"].keep(off=off, vtx=vtx), "first": state["first"]}
    if op == "serve":
        return state["requests"].burst()
    h = state["own"].handle
    if op == "host":
        n_poly, n_vtx = pg.run_host(h, state["xy"], state["tri"], None, *state["csr"])
        return {"csr": state["csr"], "n_poly": n_poly, "n_vtx": n_vtx}
    pg.mesh_build_twin(h)
    pg.trivertex(h)
    return {"twin": state["twin"], "trivertex": pg.get_trivertex(h, state["n"])}


def work(case: dict) -> dict:
    """Bytes of one pass: inputs in and outputs out, once each (n points, 2n triangles;
    per triangle about 0.16 polygons and 1.3 polygon vertices, 0.15 seeds).  Integer
    gathers and comparisons; the few operations per edge are not counted."""
    n = case["n"]
    op = case["op"]
    if op in ("batch", "serve"):  # point counts log-uniform in [lo, n]
        lo = 200 if op == "batch" else 1_000
        n = case["count"] * (n - lo) / np.log(n / lo) if n > lo else case["count"] * n
    elif case["kind"] == "holes":  # what the notch and the disks leave
        n = 0.75 * n
    m = 2 * n
    csr = 8 * 0.161 * m + 4 * 1.32 * m
    mesh_in = 16 * n + 24 * m
    total = {
        "run": mesh_in + csr + m,
        "phases": mesh_in + csr + m + 4 * 0.151 * m + 8 * 0.151 * m + 4 * 1.3 * m + 8 * m,
        "batch": mesh_in + csr + 8 * case.get("count", 0),
        "serve": mesh_in + csr,
        "host": 16 * n + 12 * m + csr,
        "twin": 12 * m + 12 * m + 4 * n,
    }[op]
    return {"bytes": float(total), "flops": 0.0}
