"""lb_adjoint's schedules: how the forward pass is cut and recorded changes neither results nor anything
else that the caller sees."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

GRID = (96, 64, 96)  # large enough for recorded advances


@pytest.fixture(scope="module")
def lb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_08923_gb300.build as b
    b.build()
    import paper_1804_08923_gb300 as lbm
    return lbm


def lattice(lb, grid=GRID, bc=(2, 3), **params):
    p = dict(dict(rho_r0=1.0, rho_b0=0.5, nu_r=0.02, nu_b=0.05, sigma=0.003, u_in=0.05, d_in=0.3 * min(grid[:2]),
                  noise_amp=0.02, seed=4, eps_grad=1e-4), **params)
    lat = lb.Lattice(grid, p, bc=bc)
    lat.init_fields(*workloads.random_two_phase_fields(grid[::-1], 3, p["rho_r0"], p["rho_b0"], u_amp=0.03))
    return lat


def test_an_adjoint_takes_no_profile_records(lb):
    lat = lattice(lb)
    lat.profile_enable(32)
    lat.adjoint(6, checkpoint=3)
    assert all(n == 0 for _, n in lat.profile_read().values())
    lat.step(3)
    assert {k: n for k, (_, n) in lat.profile_read().items() if n} == {
        "boundary_kernel": 1, "moment_kernel": 1, "advance_kernel": 2, "collide_kernel": 1}
    lat.close()
