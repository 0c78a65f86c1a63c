"""A training step in which a bounded wait gives up (injected from the host:
SBR_FAULT=timeout, a barrier that nothing arrives at) reports it and leaves the
parameters as they were; inference reports it too. The context stays usable.
"""
import os

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_failed_step_changes_no_parameter():
    import paper_2208_10006_gb300 as sbr
    g = torch.Generator(device="cuda").manual_seed(1)
    x, y = torch.rand(300, 4, device="cuda", generator=g), torch.rand(300, 6, device="cuda", generator=g)
    make = lambda: sbr.MLP(6, (0, 0, 0, 0), (1, 1, 1, 1), width=128, depth=2, max_batch=300, seed=3)
    m = make()
    m.train_step(x, y)
    m.status()
    before, grad = m.params(0).clone(), m.params(2).clone()
    os.environ["SBR_FAULT"] = "timeout"
    try:
        m.train_step(x, y)
        torch.cuda.synchronize()
    finally:
        os.environ.pop("SBR_FAULT", None)
    with pytest.raises(sbr.SbrError) as e:
        m.status()
    assert e.value.status == 5
    assert torch.equal(m.params(0), before) and torch.equal(m.params(2), grad)
    m.train_step(x, y)   # and the steps after it
    assert torch.equal(m.params(0), before)
    # another network trains as usual
    n = make()
    n.train_step(x, y)
    n.status()
    assert torch.equal(n.params(0), before)


def test_failed_prediction_is_reported():
    import paper_2208_10006_gb300 as sbr
    m = sbr.MLP(6, (0, 0, 0, 0), (1, 1, 1, 1), width=256, depth=3, max_batch=40000, seed=3)
    x = torch.rand(40000, 4, device="cuda")
    want = m.predict(x).clone()
    os.environ["SBR_FAULT"] = "timeout"
    try:
        m.predict(x)
        torch.cuda.synchronize()
    finally:
        os.environ.pop("SBR_FAULT", None)
    with pytest.raises(sbr.SbrError) as e:
        m.status()
    assert e.value.status == 5
    assert torch.equal(m.predict(x), want)
