"""The tensors that Lattice.fields returns are the caller's own: each with its storage and alignment."""
import pytest

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


@pytest.mark.parametrize("grid", [(7, 5, 9), (32, 32, 32), (41, 41, 41)])
def test_fields_are_tensors_of_their_own(lb, grid):
    import torch
    lat = lb.Lattice(grid, dict(rho_r0=1.0, rho_b0=0.5, nu_r=0.05, nu_b=0.1, sigma=0.004))
    lat.init_uniform(0.3, 0.2)
    F = lat.fields()
    assert len({t.untyped_storage().data_ptr() for t in F.values()}) == len(F) == 7
    for t in F.values():
        assert t.data_ptr() % 256 == 0 and t.is_contiguous() and t.storage_offset() == 0
        assert t.untyped_storage().nbytes() == 4 * lat.nodes
    w = torch.ones((), device="cuda", requires_grad=True)
    F["phi"].mul_(w)  # a field can enter a differentiated expression in place, alone
    assert F["phi"].requires_grad and not F["rho_r"].requires_grad
    lat.close()
