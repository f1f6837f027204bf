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


def test_step_beside_a_capture_of_another_thread(pfg, params):
    """Steps that are not waited for launch kernels only, also where a step becomes a graph, so a capture in the default
    (global) mode elsewhere in the process goes on."""
    import threading

    import torch
    y = synth.ic_spheres(32, 2, 3.0, 4.0, 3, params)
    with pfg.Simulation(y.shape[1:], params, "euler", "fp64", stream=torch.cuda.Stream()) as s, \
            pfg.Simulation(y.shape[1:], params, "euler", "fp64", stream=torch.cuda.Stream()) as ref:
        for sim in (s, ref):
            sim.set_state(y)
        for _ in range(20):  # its kernels are loaded, and those of its graph
            ref.step(0.25)
        a = torch.zeros(1000, device="cuda")
        torch.cuda.synchronize()
        err = []

        def steps():
            try:
                for _ in range(20):
                    s.step(0.25)
            except Exception as e:  # noqa: BLE001
                err.append(e)

        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            a += 1.0
            t = threading.Thread(target=steps)
            t.start()
            t.join()
            a += 1.0
        graph.replay()
        torch.cuda.synchronize()
        assert not err, err
        assert float(a[0]) == 2.0
        assert np.array_equal(s.state_hat().cpu().numpy(), ref.state_hat().cpu().numpy())


@pytest.mark.parametrize("prec,shape", [("fp32bulk", (32, 32, 32)), ("fp64", (16, 18, 20)), ("fp32bulk", (24, 20, 54))])
def test_tolerances_change_from_step_to_step(pfg, params, prec, shape):
    """More tolerances than a context keeps graphs, step by step, and step sizes that change without a wait between."""
    y = synth.random_state(shape, 5, phi_scale=0.9)
    out = []
    for direct in (True, False):
        with pfg.Simulation(shape, params, "ark3", prec) as s:
            s.set_state(y)
            s.profile(direct)
            s.set_time(0.0, 0.1)
            e = []
            for k in range(60):
                s.advance_attempts(1, 1e30, 1e-4 * (1 + k % 23), 1e-8 * (1 + k % 5))
                e += [s.attempts()[0], s.time()]
                s.set_time(0.0, 0.05 + 0.001 * (k % 7))
            out.append((s.state_hat().cpu().numpy(), e))
    assert out[0][1] == out[1][1]
    assert np.array_equal(out[0][0], out[1][0])


def test_step_sizes_that_change_unwaited(pfg, params):
    y = synth.ic_spheres(32, 2, 3.0, 4.0, 3, params)
    out = []
    for direct in (True, False):
        with pfg.Simulation(y.shape[1:], params, "euler", "fp32bulk") as s:
            s.set_state(y)
            s.profile(direct)
            for k in range(60):  # no method with an estimate: not waited for
                s.step(0.05 + 0.01 * (k % 9))
            out.append(s.state_hat().cpu().numpy())
    assert np.array_equal(out[0], out[1])


def test_context_on_a_capturing_stream(pfg, params):
    """A step on a stream under capture is refused at its wait, from the first step and after graphs were built, and the
    context steps on afterwards."""
    import ctypes

    import torch
    rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    y = synth.ic_spheres(32, 2, 3.0, 4.0, 3, params)
    st = torch.cuda.Stream()
    raw, graph = ctypes.c_void_p(st.cuda_stream), ctypes.c_void_p()
    with pfg.Simulation(y.shape[1:], params, "ark4", "fp32bulk", stream=st) as s:
        for steps in (1, 20):
            s.set_state(y)
            for _ in range(steps):
                s.step(0.25)
            torch.cuda.synchronize()
            assert rt.cudaStreamBeginCapture(raw, 1) == 0  # thread-local mode
            with pytest.raises(pfg.PFError):
                s.step(0.25)
            assert rt.cudaStreamEndCapture(raw, ctypes.byref(graph)) != 0  # the wait ended the capture
            rt.cudaGetLastError()
        s.set_state(y)
        s.step(0.25)
        got = s.state_hat().cpu().numpy()
    with pfg.Simulation(y.shape[1:], params, "ark4", "fp32bulk") as s:
        s.set_state(y)
        s.step(0.25)
        assert np.array_equal(got, s.state_hat().cpu().numpy())
