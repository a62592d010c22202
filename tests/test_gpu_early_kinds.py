"""Blocks beside the walk that have one kind of the listed seeds and not the other.

Domains with holes cut out of mixture meshes have more border terminal edges than the
blocks take, and few enough long ones: the blocks then have the long kind alone.  On these
meshes a block splits one of its regions along the region's own terminal edge while the
walk goes through the seeds; with per-kernel timing on, it has done so before the walk
begins."""
from __future__ import annotations

import functools

import numpy as np
import pytest

import meshgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2204_05438_gb300 as pg  # noqa: E402
from test_gpu_parity import unpack_labels  # noqa: E402


@functools.lru_cache(maxsize=None)
def domain(n, seed):
    """The mesh and the oracle's arrays, with what the case is made for asserted."""
    mesh = meshgen.domain_with_holes("gmm", n, 1 << 24, seed)
    ref = oracle.full(mesh)
    twin = np.asarray(mesh["twin"]).reshape(-1)
    tri, xy = np.asarray(mesh["tri"]).reshape(-1, 3), np.asarray(mesh["xy"])
    h = 3 * ref["seeds"] + ref["label"]["max_edge"][ref["seeds"]]
    d = (xy[np.roll(tri, -1, axis=1)] - xy[tri]).astype(np.int64)
    sq = (d * d).sum(axis=2).reshape(-1)
    border = twin[h] < 0
    far = ~border & (sq[h] > sq.max() // 256)  # at least a 16th of the longest edge
    assert border.sum() > 256 and 0 < far.sum() < 256
    assert ref["frontier_final"][h[far]].any(), "no terminal edge of these is a split edge"
    return mesh, ref


@pytest.mark.parametrize("timing", [True, False])
@pytest.mark.parametrize("n,seed", [(200_000, 5), (350_000, 3), (350_000, 7)])
def test_long_kind_alone_beside_the_walk(n, seed, timing):
    mesh, ref = domain(n, seed)
    M = pg.from_numpy(mesh)
    pg.set_timing(M.handle, timing)
    for phases in (False, True, False):
        if phases:
            M.label(), M.seeds(), M.traverse()
            off, vtx = (t.cpu().numpy() for t in M.polygons())
            np.testing.assert_array_equal(off, ref["trav_off"])
            np.testing.assert_array_equal(vtx, ref["trav_vtx"])
            M.repair()
        else:
            M.run()
        off, vtx = (t.cpu().numpy() for t in M.polygons())
        np.testing.assert_array_equal(off, ref["off"])
        np.testing.assert_array_equal(vtx, ref["vtx"])
        lab = unpack_labels(M.labels().cpu().numpy())
        np.testing.assert_array_equal(lab["frontier"], ref["frontier_final"])
        st = M.stats()
        assert st["n_vtx_trav"] == len(ref["trav_vtx"]) and st["n_splits"] == ref["splits"]
    M.close()
