"""The one-block forms of small inputs against the general launches: the tree of up
to 1,024 primitives (SBR_BVH_PHASES=1 keeps to a launch per phase), the order of path
keys (SBR_SORT_PHASES=1: a launch per word), and the export into device arrays against
copies to the host. Integers and FP64 values, all compared exactly.
"""
import numpy as np
import pytest
import torch

import oracle
import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sbr():
    import paper_2208_10006_gb300 as m
    return m


def _scene(T, n_rx, seed):
    rng = np.random.default_rng(seed)
    c = rng.uniform(-20, 20, (T, 1, 3))
    if T > 8:
        c[: T // 4] = c[0]          # equal Morton codes: the order falls back to the index
    tri = (c + rng.uniform(-6, 6, (T, 3, 3))).astype(np.float32)
    return dict(tri=torch.as_tensor(tri, device="cuda"), sid=torch.arange(T, dtype=torch.int32, device="cuda"), S=T,
                tx=[0.3, -0.2, 0.1], rx=torch.as_tensor(rng.uniform(-15, 15, (n_rx, 3)), device="cuda"))


def _run(sbr, d, sah=False):
    bvh = sbr.build_bvh(d["tri"], d["sid"], d["S"], sah_top=sah)
    tr = sbr.trace(bvh, d["tx"], d["rx"], 40, 2, count_visits=True, table_log2=18)
    st = tr.stats()
    pl = sbr.paths(tr, bvh)
    return bvh.info(), {k: st[k] for k in ("node_visits", "tri_tests", "rx_visits", "keys", "ray_bounces", "alpha")}, \
        {k: v.cpu().numpy() for k, v in pl.export().items()}


@pytest.mark.parametrize("T,n_rx", [(1, 1), (2, 2), (3, 33), (31, 32), (32, 1), (33, 3), (255, 64), (1023, 257), (1024, 1024),
                                    (1025, 1025)])
def test_tree_and_order_of_small_sets(sbr, monkeypatch, T, n_rx):
    d = _scene(T, n_rx, T)
    a = _run(sbr, d)
    monkeypatch.setenv("SBR_BVH_PHASES", "1")
    monkeypatch.setenv("SBR_SORT_PHASES", "1")
    b = _run(sbr, d)
    assert a[0] == b[0] and a[1] == b[1]
    assert len(a[2]["rx"]) > 0 or T == 1   # (one face may hide the one receiver)
    for k in a[2]:
        assert np.array_equal(a[2][k], b[2][k]), k


@pytest.mark.parametrize("alpha", [0.0, 0.01])
def test_alpha_of_the_launch_grid(sbr, alpha):
    d = _scene(3, 1, 5)
    bvh = sbr.build_bvh(d["tri"], d["sid"], 3)
    got = sbr.trace(bvh, d["tx"], d["rx"], 12, 1, alpha=alpha).stats()["alpha"]
    want = alpha or oracle.alpha(12)
    assert abs(got - want) <= 1e-13 * want


@pytest.mark.parametrize("shift", [0, 1, 3])
def test_export_into_unaligned_arrays(sbr, shift):
    r = sbr.run_scene(scenes.shoebox(N=60, K=3, n_rx=5))
    pl, ref = r["paths"], r["export"]
    out = {}
    for k, v in ref.items():     # device arrays that begin `shift` elements into a buffer, guarded at both ends
        buf = torch.full((v.numel() + 2 * shift + 2,), 77, dtype=v.dtype, device="cuda")
        out[k] = buf[shift: shift + v.numel()].view(v.shape)
        out["_" + k] = buf
    pl.export(out={k: out[k] for k in ref})
    host = {k: torch.empty(v.shape, dtype=v.dtype).pin_memory() for k, v in ref.items()}
    pl.export(out=host)
    torch.cuda.synchronize()
    for k, v in ref.items():
        assert torch.equal(out[k].cpu(), host[k]) and torch.equal(v.cpu(), host[k]), k
        buf = out["_" + k]
        assert (buf[:shift] == 77).all() and (buf[shift + v.numel():] == 77).all(), k
