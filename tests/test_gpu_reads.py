"""Reading a handle's results: by several threads at once, with nothing allocated, and not
under a stream capture."""
from __future__ import annotations

import ctypes
import threading

import numpy as np
import pytest

import meshgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2204_05438_gb300 as pg  # noqa: E402

OOM = 4


def test_threads_read_one_new_handle_at_once():
    mesh = meshgen.generate("gmm", 3_000, 1 << 20, 91)
    ref = oracle.run(mesh)
    for _ in range(10):
        M = pg.from_numpy(mesh)
        M.run()
        got, start = [], threading.Barrier(6)

        def read(k):
            start.wait()
            for _ in range(20):
                if k % 2:
                    got.append([t.numel() for t in M.polygons()])
                else:
                    st = M.stats()
                    got.append([st["n_poly"] + 1, st["n_vtx"]])

        threads = [threading.Thread(target=read, args=(k,)) for k in range(6)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert len(got) == 120
        assert all(g == [len(ref["off"]), len(ref["vtx"])] for g in got)
        off, vtx = (t.cpu().numpy() for t in M.polygons())
        np.testing.assert_array_equal(off, ref["off"])
        np.testing.assert_array_equal(vtx, ref["vtx"])
        M.close()


def test_phases_and_reads_allocate_nothing():
    """With the library's next allocation set to fail, a new handle's phases and first
    reads go through, and the failure is still there for the next handle."""
    mesh = meshgen.generate("uniform", 5_000, 1 << 20, 92)
    M = pg.from_numpy(mesh)
    try:
        pg.debug_fail_alloc(1)
        M.run()
        M.polygons(), M.stats(), M.seed_list()
        M.label(), M.seeds(), M.traverse(), M.repair()
        M.polygons(), M.lepp()
        with pytest.raises(pg.PolyllaError) as e:
            pg.from_numpy(mesh)
        assert e.value.code == OOM
    finally:
        pg.debug_fail_alloc(0)
    M.close()


@pytest.mark.parametrize("mode", [0, 2], ids=["global", "relaxed"])
def test_read_under_capture_is_refused(mode):
    """A read waits for the device, which a stream capture does not allow: it fails, and it
    leaves no graph behind that would write to the read's memory."""
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    mesh = meshgen.generate("uniform", 5_000, 1 << 20, 93)
    ref = oracle.run(mesh)
    M = pg.from_numpy(mesh)
    s = torch.cuda.Stream()
    M.run(s)
    M.polygons()
    at, graph = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(at, mode) == 0
    M.run(s)
    with pytest.raises(pg.PolyllaError):
        M.polygons()
    assert rt.cudaStreamEndCapture(at, ctypes.byref(graph)) != 0
    assert not graph.value
    rt.cudaGetLastError()
    M.run(s)
    off, vtx = (t.cpu().numpy() for t in M.polygons())
    np.testing.assert_array_equal(off, ref["off"])
    np.testing.assert_array_equal(vtx, ref["vtx"])
    M.close()
