"""The statistic of several-tip pieces whose smallest vertex repeats (n_multi_turn)."""
from __future__ import annotations

import numpy as np
import pytest

import meshgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2204_05438_gb300 as pg  # noqa: E402


def pieces(ref):
    """Per split polygon of the traversal: (length, tips, pieces whose smallest vertex
    repeats)."""
    to, tv, fo, fv = (ref[k] for k in ("trav_off", "trav_vtx", "off", "vtx"))
    first = 0
    for i in range(len(to) - 1):
        v = tv[to[i]:to[i + 1]]
        k = 1  # k pieces have 2 (k - 1) more vertices than the polygon, and no fewer do
        while fo[first + k] - fo[first] != len(v) + 2 * (k - 1):
            k += 1
        if k > 1:
            parts = [fv[fo[q]:fo[q + 1]] for q in range(first, first + k)]
            yield len(v), int((v == np.roll(v, -2)).sum()), sum((p == p.min()).sum() > 1 for p in parts)
        first += k


@pytest.mark.parametrize("swap,want", [(None, 0), (9141, 1)])
def test_pieces_with_a_repeated_smallest_vertex(swap, want):
    """A 40-vertex polygon with two tips has a piece that meets vertex 9141 twice; with
    the ids 0 and 9141 exchanged that is its smallest."""
    mesh = meshgen.generate("gmm", 20_000, 1 << 20, 1)
    if swap is not None:
        p = np.arange(len(mesh["xy"]))
        p[[0, swap]] = [swap, 0]
        mesh = {"xy": mesh["xy"][p], "tri": p[mesh["tri"]].astype(np.int32), "twin": mesh["twin"]}
    ref = oracle.full(mesh)
    assert sum(n for length, tips, n in pieces(ref) if length <= 64 and 2 <= tips <= 8) == want
    M = pg.from_numpy(mesh)
    M.run()
    off, vtx = (t.cpu().numpy() for t in M.polygons())
    np.testing.assert_array_equal(off, ref["off"])
    np.testing.assert_array_equal(vtx, ref["vtx"])
    assert M.stats()["n_multi_turn"] == want
    M.close()
