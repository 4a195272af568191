"""lb_step(n) from moment record to moment record (advance_kernel) against n single steps, which
gather and write the populations every step: the same bits, for every boundary and at the tile's
remainders.  The lattices are large enough for lb_step to choose the advance."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

P, S, I, C = 0, 1, 2, 3  # periodic, free slip, inlet, convective


@pytest.fixture(scope="module")
def lb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_08923_gb300.build as b
    b.build()
    import paper_1804_08923_gb300 as lbm
    return lbm


def pair(lb, grid, params, bc, seed):
    nx, ny, nz = grid
    fields = workloads.random_two_phase_fields((nz, ny, nx), seed, params["rho_r0"], params["rho_b0"], u_amp=0.03)
    out = []
    for _ in range(2):
        lat = lb.Lattice(grid, params, bc=bc)
        lat.init_fields(*fields)
        out.append(lat)
    return out


def same(a, b):
    import torch
    assert torch.equal(a.populations(), b.populations())
    assert np.array_equal(a.history(), b.history())
    assert a.step_count == b.step_count


@pytest.mark.parametrize("grid,bc", [
    ((96, 64, 96), (P, P, P, P)),   # whole tiles
    ((97, 65, 300), (P, P, P, P)),   # one node over in x, y
    ((127, 63, 150), (S, S, P, P)),  # one short
    ((100, 70, 140), (I, C, P, P)),
    ((96, 66, 150), (I, S, S, P)),
    ((125, 99, 95), (I, C, S, S)),
    ((64, 97, 150), (S, C, P, S)),
    ((70, 66, 400), (S, S, S, S)),
])
@pytest.mark.parametrize("g", [(0.0, 0.0, 0.0), (1e-6, -2e-6, 1e-5)])
def test_several_steps_equal_single_steps(lb, grid, bc, g):
    params = dict(rho_r0=1.0, rho_b0=0.4, nu_r=0.01, nu_b=0.03, sigma=0.004, g=g, u_in=0.05, d_in=0.4 * min(grid[:2]),
                  noise_amp=0.02, seed=9, fourier=(0.05, 0.02, -0.03))
    a, b = pair(lb, grid, params, bc, 3)
    for n in (2, 3, 6):  # the state ends in either buffer
        l0 = a.kernel_launches
        a.step(n)
        assert a.kernel_launches - l0 == n + 1 + (bc[0] != P), "the advance was not taken"
        for _ in range(n):
            b.step(1)
        same(a, b)
    assert np.isfinite(a.mass()).all()
    a.close()
    b.close()


@pytest.mark.parametrize("alpha_mix,s2b", [(1, 1.0), (0, 1.3)])
def test_options_of_the_collision(lb, alpha_mix, s2b):
    """alpha-bar by mass fractions, and a bulk rate away from 1 (the trace of the second moment
    relaxes too)."""
    params = dict(rho_r0=5.0, rho_b0=1.0, nu_r=0.02, nu_b=0.05, sigma=0.003, alpha_mix=alpha_mix, s2b=s2b)
    a, b = pair(lb, (96, 64, 96), params, (P, P, P, P), 5)
    a.step(5)
    for _ in range(5):
        b.step(1)
    same(a, b)


def test_mass_checks_save_and_load_between(lb):
    """check_every ends an advance at every multiple; a checkpoint taken between two calls resumes
    the same run."""
    params = dict(rho_r0=1.0, rho_b0=0.5, nu_r=0.02, nu_b=0.05, sigma=0.003, check_every=4)
    a, b = pair(lb, (96, 64, 96), params, (P, P, P, P), 6)
    a.step(3)
    blob = a.save()
    a.step(8)
    for _ in range(11):
        b.step(1)
    same(a, b)
    b.load(blob)
    b.step(8)
    same(a, b)


def test_uniform_rest_state_is_a_fixed_point_of_the_advance(lb):
    shape = (90, 66, 70)
    params = dict(rho_r0=1.0, rho_b0=2 / 3, nu_r=4e-4, nu_b=4e-4, sigma=4e-4)
    lat = lb.Lattice(shape[::-1], params, bc=(S, C))
    for rr, rb in ((0.0, 2 / 3), (0.3, 0.4)):
        lat.init_fields(np.full(shape, rr, np.float32), np.full(shape, rb, np.float32), np.zeros((3,) + shape, np.float32))
        lat.step(1)
        s1 = lat.populations().clone()
        lat.step(40)
        assert bool((lat.populations() == s1).all())
        F = lat.fields()
        assert not F["ux"].any() and not F["uy"].any() and not F["uz"].any()
