"""The twin array built on the device, at the edges of its tiles of 512 triangles.

Half-edges are paired within a tile, in a first slot or a second, or through a table
that all tiles share; each directed edge may be used once.  Expected twins come from
sorting the directed edges; they are whole numbers and must be equal."""
from __future__ import annotations

import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2204_05438_gb300 as pg  # noqa: E402

TILE = 512


def expected(tri: np.ndarray, n: int) -> np.ndarray:
    u = tri.reshape(-1).astype(np.int64)
    v = tri[:, [1, 2, 0]].reshape(-1).astype(np.int64)
    order = np.argsort(u * n + v)
    keys = (u * n + v)[order]
    at = np.minimum(np.searchsorted(keys, v * n + u), len(keys) - 1)
    return np.where(keys[at] == v * n + u, order[at], -1)


def built(xy: np.ndarray, tri: np.ndarray) -> np.ndarray:
    n, m = len(xy), len(tri)
    h = pg.mesh_create_host(n, m)
    try:
        d_xy, d_tri, d_twin = pg.mesh_inputs(h, n, m)
        d_xy.copy_(torch.as_tensor(np.ascontiguousarray(xy).reshape(-1)))
        d_tri.copy_(torch.as_tensor(np.ascontiguousarray(tri, dtype=np.int32).reshape(-1)))
        d_twin.fill_(7)
        torch.cuda.synchronize()
        pg.mesh_build_twin(h)
        torch.cuda.synchronize()
        return d_twin.cpu().numpy()
    finally:
        pg.mesh_destroy(h)


def rejected(xy: np.ndarray, tri: np.ndarray) -> int:
    with pytest.raises(pg.PolyllaError) as e:
        pg.mesh_create(torch.as_tensor(np.ascontiguousarray(xy)).cuda(),
                       torch.as_tensor(np.ascontiguousarray(tri, dtype=np.int32)).cuda(), None, 0)
    return e.value.code


def mesh(points: int = 3000):
    m = meshgen.generate("gmm", points, 1 << 20, 31)
    return np.asarray(m["xy"]).reshape(-1, 2), np.asarray(m["tri"]).reshape(-1, 3)


@pytest.mark.parametrize("m", [1, 2, TILE - 1, TILE, TILE + 1, 2 * TILE, 5 * TILE + 3])
@pytest.mark.parametrize("order", ["local", "random"])
def test_tile_edges(m, order):
    xy, tri = mesh()
    if order == "random":
        tri = np.random.default_rng(m).permutation(tri)
    tri = tri[:m]
    xy, tri = xy[np.unique(tri)], np.unique(tri, return_inverse=True)[1].reshape(-1, 3)
    np.testing.assert_array_equal(built(xy, tri), expected(tri, len(xy)))


@pytest.mark.parametrize("k", [40, 700, 9000])
@pytest.mark.parametrize("last", [False, True])
def test_fan(k, last):
    """A hub with k triangles: one vertex owns half of the edges."""
    hub, rim = (k, np.arange(k)) if last else (0, 1 + np.arange(k))
    tri = np.stack([np.full(k, hub), rim, np.roll(rim, -1)], 1)
    xy = np.stack([np.arange(k + 1), np.arange(k + 1) ** 2 % 1009], 1).astype(np.int64)
    np.testing.assert_array_equal(built(xy, tri), expected(tri, k + 1))


@pytest.mark.parametrize("gap", [1, TILE, 4 * TILE])
@pytest.mark.parametrize("what", ["triangle", "pair", "third", "same"])
def test_edges_used_twice(gap, what):
    """An edge of a triangle pair, again `gap` triangles on: in the tile or in another."""
    xy, tri = mesh()
    n = len(xy)
    tw = expected(tri, n)
    h = int(np.flatnonzero((tw >= 0) & (tw // 3 < 40) & (np.arange(len(tw)) < 120))[0])
    u, v = tri.reshape(-1)[h], tri[:, [1, 2, 0]].reshape(-1)[h]
    xy = np.concatenate([xy, xy[:2] + 1])
    more = {"triangle": [tri[h // 3]], "pair": [tri[h // 3], tri[tw[h] // 3]],
            "third": [[v, u, n]], "same": [[u, v, n]]}[what]
    at = h // 3 + gap
    assert rejected(xy, np.concatenate([tri[:at], np.asarray(more, tri.dtype), tri[at:]])) == 3


def test_pair_again_in_another_tile():
    """Both triangles of an edge in one tile, and two others on that edge in another tile:
    each tile pairs its own."""
    xy, tri = mesh()
    n = len(xy)
    tw = expected(tri, n)
    h = int(np.flatnonzero((tw >= 0) & (tw // 3 < 40) & (np.arange(len(tw)) < 120))[0])
    u, v = tri.reshape(-1)[h], tri[:, [1, 2, 0]].reshape(-1)[h]
    xy = np.concatenate([xy, xy[:2] + 1])
    assert rejected(xy, np.concatenate([tri, [[u, v, n], [v, u, n + 1]]])) == 3


def test_out_of_range_comes_first():
    xy, tri = mesh()
    bad = np.concatenate([tri, tri[:5]])
    bad[-1, 1] = len(xy)
    assert rejected(xy, bad) == 2


def test_edge_from_a_vertex_to_itself():
    tri = np.array([[0, 0, 1], [2, 3, 4]])
    xy = np.array([[0, 0], [4, 0], [9, 9], [12, 9], [10, 14]], dtype=np.int64)
    np.testing.assert_array_equal(built(xy, tri), [0, 2, 1, -1, -1, -1])
    assert rejected(xy, np.array([[0, 0, 0], [2, 3, 4]])) == 3
