"""Device memory of a context: the elastic-kernel table is taken where there is room for it."""
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
