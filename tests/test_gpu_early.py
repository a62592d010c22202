"""Regions that may be long, taken by thread blocks beside the walk.

Seeds whose terminal edge is a border edge, or at least a 16th of the mesh's longest
edge, are listed; up to 256 of either kind are the blocks', more are the walk's.  The
polygons are the same whole numbers either way: on meshes with just as many listed seeds
as the limit and one more, with none, and with regions beyond what such a block holds
(2048 triangles), in the phases and in the run."""
from __future__ import annotations

import numpy as np
import pytest

import meshgen
import oracle
from meshlib import disjoint_union, spiral_wheel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2204_05438_gb300 as pg  # noqa: E402
from test_gpu_parity import assert_parity  # noqa: E402


def strips(count: int, inner: int = 3000):
    """`count` single triangles (a border terminal edge each) beside a random mesh."""
    base = meshgen.generate("uniform", inner, 1 << 18, 41)
    n = len(base["xy"])
    k = np.arange(count)
    corner = np.stack([(1 << 20) + 64 * (k % 64), 64 * (k // 64)], 1)
    xy = np.concatenate([corner + d for d in ([0, 0], [40, 0], [0, 30])])
    tri = np.stack([k, k + count, k + 2 * count], 1) + n
    return {"xy": np.concatenate([base["xy"], xy]).astype(np.int64),
            "tri": np.concatenate([base["tri"], tri]).astype(np.int32),
            "twin": np.concatenate([np.asarray(base["twin"]).reshape(-1),
                                    np.full(3 * count, -1)]).astype(np.int32)}


def border_seeds(mesh) -> int:
    lab = oracle.full(mesh)["label"]
    k, seed = (np.asarray(lab[x]).reshape(-1) for x in ("max_edge", "seed"))
    twin = np.asarray(mesh["twin"]).reshape(-1)
    return int(((twin[3 * np.arange(len(k)) + k] < 0) & (seed != 0)).sum())


@pytest.mark.parametrize("over", [-1, 0, 1, 40])
def test_listed_seeds_about_the_limit(over):
    here = border_seeds(strips(1)) - 1
    mesh = strips(256 + over - here)
    assert border_seeds(mesh) == 256 + over
    assert_parity(mesh)


@pytest.mark.parametrize("m", [8191, 8192, 8193, 12288, 12289])
def test_tiles_of_the_seed_pass(m):
    """Sizes about whole tiles of 4096 triangles."""
    mesh = strips(m - len(strips(1)["tri"]) + 1)
    assert len(mesh["tri"]) == m
    assert_parity(mesh)


@pytest.mark.parametrize("k", [63, 64, 500, 2045, 2046, 2047, 2100])
def test_long_regions_beside_the_walk(k):
    """Wheels of k triangles: about the walk's limit, and about what a block holds."""
    g = assert_parity(disjoint_union([meshgen.generate("uniform", 2000, 1 << 22, 42),
                                      spiral_wheel(k)]))
    assert g["stats"]["n_long"] >= (k >= 64)


@pytest.mark.parametrize("kind,n", [("gmm", 60_000), ("uniform", 150_000)])
def test_repeated_runs_and_phases(kind, n):
    mesh = meshgen.generate(kind, n, 1 << 24, 43)
    ref = oracle.run(mesh)
    M = pg.from_numpy(mesh)
    for k in range(4):
        if k == 2:  # a traversal in between lists anew and walks twice
            M.label(), M.seeds(), M.traverse(), M.repair()
        else:
            M.run()
        off, vtx = (t.cpu().numpy() for t in M.polygons())
        np.testing.assert_array_equal(off, ref["off"])
        np.testing.assert_array_equal(vtx, ref["vtx"])
    M.close()
