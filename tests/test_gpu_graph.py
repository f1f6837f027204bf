"""Steps that run as a graph (contexts that have stepped on) against the same
steps launched one kernel at a time (a context whose profiler is on): bitwise
equal states, error norms and step sizes."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pfg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_36100_gb300 as m
    m.build()
    return m


@pytest.mark.parametrize("method,prec", [("ark4", "fp32bulk"), ("ark4", "fp64"), ("ark3", "fp32bulk"),
                                         ("euler", "fp64"), ("euler", "fp32bulk")])
def test_graph_steps_equal_direct_steps(pfg, params, method, prec):
    import torch
    y = synth.ic_spheres(32, 2, 3.0, 4.0, 3, params)
    out = []
    for direct in (True, False):
        with pfg.Simulation(y.shape[1:], params, method, prec) as s:
            s.set_state(y)
            s.profile(direct)
            e = []
            for k in range(40):  # two step sizes, with and without the estimate, not waited for between
                e.append(s.step(0.25 if k % 5 else 0.125, want_lte=k % 3 != 0))
            if method != "euler":
                s.set_time(0.0, 0.25)
                for rtol in (1e-4, 1e-5, 1e-4):
                    s.advance_attempts(9, 1e30, rtol, 1e-8)
                    e += [a[2] for a in s.attempts()] + [s.time()[1]]
            cfg = s.tuning()
            cfg[1] = 8
            s.set_tuning(cfg)  # graphs of the old schedule are dropped
            for _ in range(5):
                e.append(s.step(0.25))
            torch.cuda.synchronize()
            out.append((s.state_hat().cpu().numpy(), e))
    assert out[0][1] == out[1][1]
    assert np.array_equal(out[0][0], out[1][0])
