"""The reverse step's kernels work on tiles of 32 x 4 columns that march chunks of planes; how a lattice
is cut depends on its extents.  A state repeated along x and y has the repeated adjoint, and every node's
arithmetic is the same wherever its tile and chunk begin, so the adjoint of the repeated lattice equals
the small one's bit for bit: tile edges, remainders of tiles and chunks against the wrap-around."""
import numpy as np
import pytest

import workloads

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


@pytest.mark.parametrize("grid,rep", [((8, 6, 20), (9, 7)),      # 72 x 42: two and a half tiles, ragged in y
                                      ((33, 5, 9), (2, 2)),      # one node beyond a tile
                                      ((31, 3, 37), (1, 3)),     # one short of a tile
                                      ((16, 4, 70), (20, 20)),   # whole tiles, long chunks against single planes
                                      ((1, 1, 5), (40, 9)),      # every neighbour is the node itself
                                      ((10, 4, 3), (13, 11))])
@pytest.mark.parametrize("bc", [(0, 0), (1, 1)])
def test_adjoint_of_a_repeated_state_is_the_repeated_adjoint(lb, grid, rep, bc):
    import torch
    nx, ny, nz = grid
    params = dict(workloads.CONFIGS["droplet32"]["params"], rho_r0=1.0, rho_b0=0.5, nu_r=0.02, nu_b=0.05, sigma=0.004,
                  g=(0.0, 0.0, 2e-5))
    fields = workloads.random_two_phase_fields((nz, ny, nx), 5, 1.0, 0.5, u_amp=0.03)
    out = []
    for rx, ry in ((1, 1), rep):
        lat = lb.Lattice((nx * rx, ny * ry, nz), params, bc=bc)
        lat.init_fields(*[np.tile(f, (1, ry, rx)) for f in fields])
        J, grad = lat.adjoint(3, "area", (1e-3,))
        out.append((J, np.asarray(grad), lat.adjoint_state(device=True).clone()))
    n = rep[0] * rep[1]
    (J0, g0, s0), (J1, g1, s1) = out
    assert torch.equal(s0.repeat(1, 1, 1, rep[1], rep[0]), s1)
    assert abs(J1 - n * J0) <= 1e-5 * abs(n * J0)
    assert np.abs(g1 - n * g0).max() <= 1e-4 * np.abs(n * g0).max()
