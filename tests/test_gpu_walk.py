"""The walk's limits: the triangle queue and the tip list of a warp, the longest walked
polygon, partly filled warps and blocks.

A warp walks 32 seeds through one queue (288 triangles, 64 passes) and one tip list (48
entries); polygons of more than 64 vertices go to the block kernel.  Hand-built regions
(tests/meshlib.py) put those limits to the test; the traversal and the final polygons
must equal the oracle's bit for bit, on the multi-kernel path."""
from __future__ import annotations

import numpy as np
import pytest

import meshgen
import oracle
from meshlib import disjoint_union, grid_mesh, spiral_wheel, tip_hub, tip_order_meshes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2204_05438_gb300 as pg  # noqa: E402


def side_by_side(meshes):
    """disjoint_union in rows of 16 (coordinates stay below 2^30)."""
    rows = [disjoint_union(meshes[i:i + 16]) for i in range(0, len(meshes), 16)]
    return disjoint_union(rows, shift=(0, 1 << 25))


def small():
    return meshgen.generate("gmm", 400, 1 << 20, 3)


CASES = {
    # regions of 61, 62, 63 triangles (63, 64, 65 boundary vertices: the last too long)
    "lengths-about-the-limit": lambda: [spiral_wheel(k) for k in (61, 62, 63, 60, 64)] * 3,
    # 32 regions of 62 triangles: the queue overflows at 32, 16 and 8 seeds a warp
    "queue-overflow": lambda: [spiral_wheel(62)] * 32 + [small()],
    # one region in the warp larger than the queue, among small ones
    "region-above-the-queue": lambda: [small(), spiral_wheel(400), small(), spiral_wheel(5000)],
    # 288 and 290 triangles in a warp's first 32 seeds: at the queue's end
    "queue-full": lambda: [spiral_wheel(9)] * 32 + [spiral_wheel(9)] * 31 + [spiral_wheel(11)],
    # ten-tip polygons side by side: more tips than a warp's list holds
    "tip-list-overflow": lambda: [tip_hub()] * 6 + [small()],
    # seed counts about a warp's, a block's and the output tiles' (256 and 1024)
    **{f"squares-{k}x{k}": (lambda k=k: [grid_mesh(k, seed=k)[0]]) for k in (1, 5, 6, 16, 17, 32, 33)},
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_walk_limits(name):
    mesh = side_by_side(CASES[name]())
    ref = oracle.full(mesh)
    M = pg.from_numpy(mesh)
    M.set_one_block(0)
    for phases in (False, True):
        if phases:
            M.label()
            M.seeds()
            M.traverse()
            off, vtx = (t.cpu().numpy() for t in M.polygons())
            np.testing.assert_array_equal(off, ref["trav_off"])
            np.testing.assert_array_equal(vtx, ref["trav_vtx"])
            M.repair()
        else:
            M.run()
        off, vtx = (t.cpu().numpy() for t in M.polygons())
        np.testing.assert_array_equal(off, ref["off"])
        np.testing.assert_array_equal(vtx, ref["vtx"])
        st = M.stats()
        assert st["n_vtx_trav"] == len(ref["trav_vtx"])
        assert st["n_splits"] == len(ref["off"]) - len(ref["trav_off"])
    M.close()


@pytest.mark.parametrize("cap", [16, 32, 48, 64])
def test_walk_cap_of_a_schedule(cap):
    """Batches walk polygons of at most the schedule's cap; the rest go to blocks."""
    meshes = [spiral_wheel(k) for k in (cap - 3, cap - 2, cap - 1, 40, 62)] + [small(), tip_hub()]
    cat = meshgen.concat(meshes)
    B = pg.batch_from_numpy(cat)
    refs = [oracle.run(m) for m in meshes]
    for k in range(pg.batch_schedules()):
        if pg.batch_schedule_info(k)["walk_cap"] != cap:
            continue
        B.run(k)
        off, vtx, first = (t.cpu().numpy().copy() for t in B.all_polygons())
        for j, ref in enumerate(refs):
            o = off[int(first[j]):int(first[j + 1]) + 1]
            np.testing.assert_array_equal(o - o[0], ref["off"], err_msg=f"schedule {k} mesh {j}")
            np.testing.assert_array_equal(vtx[o[0]:o[-1]] - cat["vtx_off"][j], ref["vtx"],
                                          err_msg=f"schedule {k} mesh {j}")
    B.close()


def test_endless_turn_on_the_multi_kernel_path_ends_with_limit_error():
    """The corrupt one-triangle mesh of test_gpu_paths.py through the kernels: it has
    no seed, so no walk meets its endless turn; the vertices that the walks found do
    not add up to the frontier half-edges, and the check of every turn reports it."""
    mesh = {"xy": np.array([[0, 0], [10, 0], [5, 1]], np.int64),
            "tri": np.array([[0, 1, 2]], np.int32), "twin": np.array([2, -1, -1], np.int32)}
    M = pg.from_numpy(mesh, validate=False)
    M.set_one_block(0)
    M.run()
    with pytest.raises(pg.PolyllaError) as e:
        M.polygons()
    assert e.value.code == 6  # POLYLLA_ERR_LIMIT
    M.close()


def test_polygons_handed_between_blocks_count_once():
    """A polygon that fits a small block (128 or 512 members) until its split edges are
    added is handed to a large one; the traversal's vertex count stays the oracle's."""
    meshes = [spiral_wheel(k) for k in (125, 126, 127, 128, 508, 509, 510, 511)] + [tip_hub()] * 3
    want = sum(len(oracle.full(m)["trav_vtx"]) for m in meshes)
    B = pg.batch_from_numpy(meshgen.concat(meshes))
    for k in range(pg.batch_schedules()):
        B.run(k)
        B.all_polygons()
        assert B.stats()["n_vtx_trav"] == want, f"schedule {k}"
    B.close()


@pytest.mark.parametrize("big", [False, True])
@pytest.mark.parametrize("rare", [False, True])
def test_several_tip_polygons(big, rare):
    """Polygons of 2 to 8 tips, split by a warp: mixture meshes (above 2^16 triangles and
    below), the meshes on which the order of the tips matters, and hubs with more tips
    than a warp takes; with every successor found by turning when `rare`."""
    meshes = tip_order_meshes() + [tip_hub(), meshgen.generate("gmm", 40_000 if big else 8_000,
                                                                1 << 22, 51)]
    mesh = side_by_side([m["mesh"] if "mesh" in m else m for m in meshes])
    ref = oracle.run(mesh)
    M = pg.from_numpy(mesh)
    M.set_one_block(0)
    pg.debug_rare_paths(M.handle, rare)
    M.run()
    off, vtx = (t.cpu().numpy() for t in M.polygons())
    lab = M.labels().cpu().numpy()
    st = M.stats()
    M.close()
    np.testing.assert_array_equal(off, ref["off"])
    np.testing.assert_array_equal(vtx, ref["vtx"])
    np.testing.assert_array_equal((lab[:, None] >> np.arange(2, 5)) & 1,
                                  ref["frontier"].reshape(-1, 3))
    assert st["n_multi_tip"] > 20 and st["n_splits"] == ref["splits"]
