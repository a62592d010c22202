"""A listed seed whose region cannot be walked (a corrupt, unvalidated mesh): the block
that has it beside the walk reports the error and leaves no polygon, neither one of an
earlier run nor one of the memory's former contents, for the output pass to copy."""
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

LIMIT = 6


def test_no_polygon_of_a_region_with_an_error():
    """Three single triangles T, S, Z beside a mesh.  A twin entry of T leads into S, whose
    longest edge leads on into Z: T's region is T and S, and a turn in S leaves it."""
    base = meshgen.generate("uniform", 3000, 1 << 18, 45)
    n, m = len(base["xy"]), len(base["tri"])
    k = np.arange(3)
    corner = np.stack([(1 << 20) + 64 * k, 0 * k], 1)  # longest edge: the second, (40,0)-(0,30)
    xy = np.concatenate([base["xy"]] + [corner + d for d in ([0, 0], [40, 0], [0, 30])])
    tri = np.concatenate([base["tri"], np.stack([k, k + 3, k + 6], 1) + n])
    twin = np.concatenate([np.asarray(base["twin"]).reshape(-1), np.full(9, -1)])
    mesh = {"xy": xy.astype(np.int64), "tri": tri.astype(np.int32), "twin": twin.astype(np.int32)}
    ref = oracle.run(mesh)
    before = len(ref["off"]) - 1 - 3  # polygons of the mesh beside
    M = pg.from_numpy(mesh)
    M.set_one_block(0)
    M.run()
    off, _ = M.polygons()
    np.testing.assert_array_equal(off.cpu().numpy(), ref["off"])
    t, s, z = 3 * (m + k)
    M.twin[t] = int(s) + 1  # T's first edge into S, by S's longest
    M.twin[s + 1] = int(z)  # and that one into Z
    torch.cuda.synchronize()
    M.run()
    with pytest.raises(pg.PolyllaError) as e:
        M.polygons()
    assert e.value.code == LIMIT
    got = off.cpu().numpy()  # the same buffer: mesh, T without vertices, Z (S has no seed)
    np.testing.assert_array_equal(got[:before + 1], ref["off"][:before + 1])
    np.testing.assert_array_equal(np.diff(got[before:before + 3]), [0, 3])
    M.close()


@pytest.mark.parametrize("edge", ["longest", "other"])
def test_twin_out_of_range_is_a_border_to_every_kernel(edge):
    """A twin one past the last half-edge, not validated: the label pass reports it and
    marks the edge frontier, so that no later kernel follows it."""
    mesh = meshgen.generate("uniform", 3000, 1 << 18, 46)
    ref = oracle.full(mesh)
    m = len(mesh["tri"])
    twin = np.asarray(mesh["twin"]).reshape(-1, 3)
    t = int(np.nonzero((twin >= 0).all(axis=1))[0][5])  # an interior triangle
    k = (int(ref["label"]["max_edge"][t]) + (edge == "other")) % 3
    M = pg.from_numpy(mesh)
    M.set_one_block(0)
    M.twin.view(-1)[3 * t + k] = 3 * m
    torch.cuda.synchronize()
    M.label()
    assert int(M.labels()[t]) >> (2 + k) & 1
    M.seeds(), M.traverse(), M.repair()
    with pytest.raises(pg.PolyllaError) as e:
        M.polygons()
    assert e.value.code == 2  # POLYLLA_ERR_RANGE
    M.close()
