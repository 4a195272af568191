"""The reverse step beside side walls, on planes of several tiles of either width (16 x 8 and 32 x 4 columns) with
ragged edges, against the oracle's complex-step tangent; and chunks of planes beside walls against
single planes."""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_adjoint import NAMES, TOL, check_components, full_params, oracle_J, tangent_gradient

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_08923_gb300.build as b
    b.build()
    import paper_1804_08923_gb300 as lbm
    return lbm


def mixture(shape):
    """Both colours and gradients of them everywhere, at the walls too (a blob that ends before the walls leaves
    their columns' sensitivities at the rounding of the others')."""
    z, y, x = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    w = lambda a, b, c, q: np.sin(2 * np.pi * (a * x + b * y + c * z) + q)
    phi = 0.45 * w(1.3, 0.7, 0.4, 0.3) + 0.3 * w(-0.8, 1.6, 0.9, 1.1)
    u = 0.03 * np.stack([w(0.6, 1.2, 0.3, 0.5), w(1.1, -0.7, 0.8, 2.0), w(0.4, 0.9, -1.2, 4.0)])
    return [np.ascontiguousarray(f, dtype=np.float32) for f in (0.5 * (1 + phi), 0.25 * (1 - phi), u)]


@pytest.mark.parametrize("nx,ny,nz", [(41, 38, 10), (66, 10, 12)])  # 3 x 5 tiles of 16 x 8, 3 x 3 of 32 x 4
@pytest.mark.parametrize("bc", [(1, 1, 1, 0), (1, 1, 0, 1), (0, 0, 1, 1)])
def test_state_gradient_on_several_walled_tiles(lb, nx, ny, nz, bc):
    """dJ/dS(0) along random directions: of all populations, and of those of the two columns at each side.
    A direction's derivative is a sum of terms of either sign; the bar is that of the repository's adjoint
    tests against the size such a sum has, |dJ/dS| |dS| over the root of the number of terms."""
    shape = (nz, ny, nx)
    params = dict(rho_r0=1.0, rho_b0=0.5, nu_r=0.02, nu_b=0.05, sigma=0.004, g=(1e-5, -2e-5, 3e-5))
    fields = mixture(shape)
    lat = lb.Lattice((nx, ny, nz), params, bc=bc)
    lat.init_fields(*fields)
    T = 4
    lat.adjoint(T, "area", (1e-3,))
    lS = lat.adjoint_state().astype(np.float64)
    ref = oracle.Lattice(oracle.make_grid(nx, ny, nz, *bc), oracle.make_params(full_params(params)))
    ref.init_fields(*fields)
    dS = np.random.default_rng(6).standard_normal((2, 27) + shape) * 1e-3
    sides = np.zeros((ny, nx))
    sides[:, [0, 1, -2, -1]] = 1.0
    sides[[0, 1, -2, -1]] = 1.0
    for d in (dS, dS * sides):
        _, tan = oracle.tangent_objective(oracle.make_grid(nx, ny, nz, *bc), full_params(params), ref.S, ref.hist, T,
                                          "area", (1e-3,), dS=d)
        ad = float((lS * d).sum())
        size = 1e-3 * np.linalg.norm(lS[d != 0])
        assert abs(ad - tan) < TOL * size, (ad, tan, size)


@pytest.mark.parametrize("nx,ny,nz,D", [(41, 38, 24, 37), (66, 10, 24, 9)])
def test_parameter_gradients_of_a_walled_jet_on_several_tiles(lb, nx, ny, nz, D):
    """An inlet disc that reaches to the walls."""
    cfg = workloads.scaled_jet("jet64", nx, ny, nz, D=D)
    params = dict(cfg["params"], noise_amp=0.02, fourier=tuple(0.05 * np.random.default_rng(5).standard_normal(16)))
    grid, bc = (nx, ny, nz), tuple(cfg["bc"]) + (1, 1)
    init = lambda r: r.init_jet()
    T, names = 6, ("u_in", "sigma", "nu_b", "a1", "b2")
    lat = lb.Lattice(grid, params, bc=bc)
    lat.init_jet()
    J, g = lat.adjoint(T, "area", (1e-3,))
    g_tan = tangent_gradient(grid, bc, params, init, T, "area", (1e-3,), names)
    J_ref = oracle_J(grid, bc, params, init, T, "area", (1e-3,))
    assert abs(J / J_ref - 1) < 1e-5, (J, J_ref)
    got = np.array([g[NAMES.index(n)] for n in names])
    assert np.abs(got - g_tan).max() / np.abs(g_tan).max() < TOL, (got, g_tan)
    check_components(got, g_tan, names)


@pytest.mark.parametrize("grid,rep", [((41, 38, 5), 64), ((66, 10, 7), 90)])
def test_chunks_of_planes_beside_walls(lb, grid, rep):
    """A state repeated along a periodic z.  With five periods a block marches one plane, with rep many,
    from every phase of the period.  The area leaves out the end planes, which three reverse steps carry
    nine planes inwards; periods further in have the same adjoint, bit for bit."""
    import torch
    nx, ny, nz = grid
    params = dict(rho_r0=1.0, rho_b0=0.5, nu_r=0.02, nu_b=0.05, sigma=0.004, g=(1e-5, -2e-5, 3e-5))
    fields = mixture((nz, ny, nx))
    states = []
    for r in (5, rep):
        lat = lb.Lattice((nx, ny, nz * r), params, bc=(0, 0, 1, 1))
        lat.init_fields(*[np.tile(f, (1,) * (f.ndim - 3) + (r, 1, 1)) for f in fields])
        lat.adjoint(3, "area", (1e-3,))
        states.append(lat.adjoint_state(device=True).clone())
        lat.close()
    period = states[0][:, :, 2 * nz:3 * nz]
    assert bool((period != 0).any())
    for k in range(2, rep - 2):
        assert torch.equal(states[1][:, :, k * nz:(k + 1) * nz], period), k


def test_long_horizon_with_checkpoints_against_the_tangent(lb):
    """100 steps of a 24x24x48 jet (D = 8, inlet noise and profile, convective outflow) in 10 segments of 10, the
    last recorded by the forward pass, the others recomputed on the second stream: J and six gradients
    against the oracle's complex-step tangent, each component against its own value."""
    cfg = workloads.scaled_jet("jet64", 24, 24, 48, D=8)
    params = dict(cfg["params"])
    params["noise_amp"] = 0.02
    params["fourier"] = tuple(0.05 * np.random.default_rng(5).standard_normal(16))
    grid, bc, T = (24, 24, 48), cfg["bc"], 100
    lat = lb.Lattice(grid, params, bc=bc)
    lat.init_jet()
    J, g = lat.adjoint(T, "area", (1e-3,), checkpoint=10)
    names = ("u_in", "sigma", "nu_r", "nu_b", "a1", "b2")
    g_tan = tangent_gradient(grid, bc, params, lambda r: r.init_jet(), T, "area", (1e-3,), names)
    J_ref = oracle_J(grid, bc, params, lambda r: r.init_jet(), T, "area", (1e-3,))
    assert abs(J / J_ref - 1) < 1e-5, (J, J_ref)
    got = np.array([g[NAMES.index(n)] for n in names])
    assert np.abs(got - g_tan).max() / np.abs(g_tan).max() < TOL, (got, g_tan)
    check_components(got, g_tan, names)
