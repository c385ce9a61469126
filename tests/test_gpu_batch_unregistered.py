"""js_batch_step_vjp takes its states per call, so a batch whose states were never registered
(js_batch_set_states) reverses a step like one whose states were."""
import numpy as np
import pytest

import oracle as O
from paper_2601_04400_gb300 import workloads as W
from jsutil import to_dev

pytestmark = pytest.mark.gpu


def test_reverse_without_registered_states():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04400_gb300 import binding as B
    probs = [W.riemann2d(40, ny=30), W.shock_cylinder(nx=64, ny=48)]
    rng = np.random.default_rng(2)
    U = [O.prim_to_cons(p, W.random_state(p, seed=3, amp=0.02)) for p in probs]
    dts = [0.4 * O.max_dt(p, u, 0.5) for p, u in zip(probs, U)]
    lam = [to_dev(rng.standard_normal(u.shape)) for u in U]
    res = []
    for register in (False, True):
        b = B.Batch(probs)
        states = [to_dev(u) for u in U]
        if register:
            b.set_states([x.clone() for x in states])
        out = [torch.empty_like(x) for x in states]
        pb = [torch.zeros(20, dtype=torch.float64, device="cuda") for _ in states]
        b.step_vjp(states, dts, lam, out, pb)
        assert b.status() == 0
        res.append((out, pb))
        b.close()
    for k in range(len(probs)):
        assert torch.equal(res[0][0][k], res[1][0][k])
        assert torch.equal(res[0][1][k], res[1][1][k])
