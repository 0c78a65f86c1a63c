"""The FP32 test ahead of a batched job's exact reception test: it may only reject what
the exact one rejects, so a batch keeps every path of the single trace (which reaches
the exact test through the receiver tree), near the origin and far from it, with
spheres from centimetres to the size of the room.
"""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sbr():
    import paper_2208_10006_gb300 as m
    return m


@pytest.mark.parametrize("shift", [0.0, 50.0, 3e3])
@pytest.mark.parametrize("N,K", [(3, 2), (12, 4), (60, 3), (200, 1)])
def test_batch_keeps_the_paths_of_the_single_trace(sbr, shift, N, K):
    sc = scenes.shoebox(N=N, K=K, n_rx=4)
    off = shift * np.array([1.0, -1.0, 0.1])
    tri = torch.as_tensor((np.asarray(sc["tri"], np.float64).reshape(-1, 3, 3) + off).astype(np.float32), device="cuda")
    sid = torch.as_tensor(sc["surface_id"], dtype=torch.int32, device="cuda")
    mats = torch.as_tensor(sc["materials"], dtype=torch.float64, device="cuda")
    bvh = sbr.build_bvh(tri, sid, len(sc["materials"]))
    f = torch.full((1,), 60e9, dtype=torch.float64, device="cuda")
    jobs = []
    for r in sc["rx"]:
        el = lambda p: torch.as_tensor(np.asarray(p)[None] + 0.0, dtype=torch.float64, device="cuda")
        tx, rx = np.asarray(sc["tx"]) + off, np.asarray(r) + off
        jobs.append(dict(scene=0, N=N, K=K, tx=tx, rx=rx, pol="V", freqs=f, gamma=torch.zeros(1, device="cuda"),
                         tx_elem=el(tx), rx_elem=el(rx)))
    b = sbr.batch_create([(bvh, mats)], jobs, config=dict(path_cap=512))
    b.run()
    n, status, _ = b.query()
    assert (status == 0).all()
    total = 0
    for i, j in enumerate(jobs):
        rx = torch.as_tensor(j["rx"][None], device="cuda")
        tr = sbr.trace(bvh, j["tx"], rx, N, K)
        pl = sbr.paths(tr, bvh)
        total += pl.n
        assert n[i] == pl.n, (i, n[i], pl.n)
        a, e = b.export(i, int(n[i])), pl.export()
        for k in ("seq", "face", "ray"):
            assert torch.equal(a[k], e[k]), (i, k)
    assert total > 4
