"""Populations read out in the canonical layout (split_kernel for FP32 storage, canonical_kernel for the
half-precision ones): device and host read-outs agree bit for bit, their sums are the densities, and a
state repeated along x and y has the repeated populations, at the remainders of the kernels' blocks."""
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


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("grid,rep", [((1, 1, 1), (2, 3)), ((5, 3, 2), (7, 1)), ((33, 9, 5), (1, 2)), ((31, 7, 6), (2, 1)),
                                      ((32, 8, 4), (1, 1)), ((16, 1, 65), (2, 9))])
def test_populations_read_out(lb, grid, rep, storage):
    import torch
    nx, ny, nz = grid
    params = dict(rho_r0=1.0, rho_b0=0.5, nu_r=0.02, nu_b=0.05, sigma=0.004, storage=storage)
    fields = workloads.random_two_phase_fields((nz, ny, nx), 4, 1.0, 0.5, u_amp=0.03)
    out = []
    for rx, ry in ((1, 1), rep):
        lat = lb.Lattice((nx * rx, ny * ry, nz), params)
        lat.init_fields(*[np.tile(f, (1, ry, rx)) for f in fields])
        lat.step(1)
        d = lat.populations(device=True).clone()
        assert np.array_equal(d.cpu().numpy(), lat.populations(device=False))
        out.append(d)
    assert torch.equal(out[0].repeat(1, 1, 1, rep[1], rep[0]), out[1])
    f = lat.fields()
    rho = torch.stack([torch.as_tensor(f["rho_r"]), torch.as_tensor(f["rho_b"])]).to(out[1].device)
    assert (out[1].sum(1) - rho).abs().max().item() <= 27 * 2.0 ** -23  # a sum of 27 numbers below 1
