"""Device memory of a context: the elastic-kernel table is taken where there is room for it, and the phase-dependent
stiffness takes 33 real fields."""
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


def free_bytes():
    import gc

    import torch
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("fp32bulk", 1e-6)])
def test_context_without_room_for_the_elastic_table(pfg, params, prec, tol):
    import torch
    n = 192
    shape = (n, n, n)
    y = synth.ic_spheres(n, 4, 3.0, 5.0, 2, params)
    table = 6 * (n // 2 + 1) ** 3 * (8 if prec == "fp64" else 4)
    with pfg.Simulation(shape, params, "euler", prec) as s:
        s.set_state(y)
        s.step(0.25)
        ref = s.get_state()
    before = free_bytes()
    with pfg.Simulation(shape, params, "euler", prec) as s:
        size = before - free_bytes()
    hold = torch.empty(free_bytes() - (size - table // 2), dtype=torch.uint8, device="cuda")
    try:
        with pfg.Simulation(shape, params, "euler", prec) as s:  # fits without the table
            s.set_state(y)
            s.step(0.25)
            got = s.get_state()
    finally:
        del hold
        free_bytes()
    for f in range(4):
        assert np.linalg.norm(got[f] - ref[f]) <= tol * np.linalg.norm(ref[f])


@pytest.mark.parametrize("prec", ["fp64", "fp32bulk"])
def test_phase_dependent_stiffness_buffers(pfg, params, prec):
    n = 128
    p = dict(params, eps_star=[[0.0] * 6] * 3)
    q = dict(params, el_inhom=1, C11_v=325.0, C12_v=176.0, C44_v=144.0)
    with pfg.Simulation((n, n, n), p, "euler", prec):
        pass
    size = []
    for r in (p, q):
        before = free_bytes()
        with pfg.Simulation((n, n, n), r, "euler", prec):
            size.append(before - free_bytes())
    # 33 fields of real points, 12 of them as half spectra (n + 2 in n), and a share of the driver's 2 MB pages
    assert size[1] - size[0] <= 36 * 8 * n ** 3
