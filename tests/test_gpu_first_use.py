"""A new handle's first run, on a busy device and on another stream than its creation.

A handle clears its look-back words, counters and stamps when it is created; a clear
that is only enqueued may run after kernels of the first run on a non-blocking stream
have begun, and take their words from under them.  Servers are created and given a
burst at once, while another stream keeps the device busy, and every result must equal
the oracle's."""
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


def test_burst_on_a_new_server():
    sizes = (900, 3_000, 9_000, 20_000, 45_000, 30_000, 6_000, 2_500)
    meshes = [meshgen.generate("gmm" if k % 2 else "uniform", n, 1 << 22, 70 + k)
              for k, n in enumerate(sizes)]
    refs = [oracle.run(m) for m in meshes]
    args = [[torch.as_tensor(m[k]).to(dt).pin_memory() for k, dt in
             (("xy", torch.int64), ("tri", torch.int32), ("twin", torch.int32))] for m in meshes]
    busy = torch.zeros(1 << 26, device="cuda")
    for _ in range(4):
        S = pg.Server(8 << 30, max_slots=12)
        for _ in range(40):
            busy.add_(1)
        ids = [S.submit(*a) for a in args * 2]
        got = {}
        while len(got) < len(ids):
            for r in S.poll(wait_us=1000):
                assert r["status"] == 0, pg.status_str(r["status"])
                got[r["id"]] = r
        for k, i in enumerate(ids):
            ref = refs[k % len(refs)]
            np.testing.assert_array_equal(got[i]["off"].numpy(), ref["off"])
            np.testing.assert_array_equal(got[i]["vtx"].numpy(), ref["vtx"])
        S.close()


def test_first_run_on_another_stream():
    mesh = meshgen.generate("gmm", 60_000, 1 << 22, 81)
    ref = oracle.run(mesh)
    dev = [torch.as_tensor(mesh[k]).to("cuda", dt).contiguous() for k, dt in
           (("xy", torch.int64), ("tri", torch.int32), ("twin", torch.int32))]
    busy = torch.zeros(1 << 26, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(6):
        for _ in range(40):
            busy.add_(1)
        M = pg.Mesh(*dev, validate=False)
        M.run(side)
        off, vtx = M.polygons()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(off.cpu().numpy(), ref["off"])
        np.testing.assert_array_equal(vtx.cpu().numpy(), ref["vtx"])
        M.close()
