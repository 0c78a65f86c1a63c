"""Traversal nodes (centre and half extent): the paths of a room far from the
origin, where FP32 centres round by more than thin boxes are wide, of scenes of one
to a few faces, and of rays along the axes, against the oracle. The FP32 walk only
culls, so the set of paths is the oracle's exactly.
"""
import numpy as np
import pytest

import oracle
import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sbr():
    import paper_2208_10006_gb300 as m
    return m


def _same_paths(sbr, sc):
    r = sbr.run_scene(sc)
    ex = {k: v.cpu().numpy() for k, v in r["export"].items()}
    o = oracle.run(sc)["paths"]
    rows = lambda p: sorted((int(p["rx"][i]), tuple(int(x) for x in p["seq"][i][: p["nb"][i]])) for i in range(len(p["rx"])))
    assert rows(ex) == rows(o)
    return len(ex["rx"])


@pytest.mark.parametrize("shift", [0.0, 1e3, 3e4])
@pytest.mark.parametrize("axes", [(1.0, 1.0, 1.0), (1.0, -1.0, 1e-3)])
def test_room_away_from_the_origin(sbr, shift, axes):
    sc = scenes.shoebox(N=40, K=2)
    off = shift * np.asarray(axes)
    for k in ("tri", "tx", "rx"):
        a = np.asarray(sc[k])
        sc[k] = (a.astype(np.float64) + off).astype(a.dtype)
    assert _same_paths(sbr, sc) > 5


@pytest.mark.parametrize("n", [1, 2, 3, 5])
def test_few_faces(sbr, n):
    sc = scenes.shoebox(N=40, K=2)
    sc["tri"], sc["surface_id"] = sc["tri"][:n], sc["surface_id"][:n]
    assert _same_paths(sbr, sc) >= 1
