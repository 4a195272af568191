"""Read-outs of an FP32 state sum a node's densities in the order in which the collision (and the initial
state) took the rest population as their remainder: fl(fl(rho - s) + s) = rho wherever the moving
populations hold between half and all of a colour's mass, which both densities here do."""
import numpy as np
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


PARAMS = dict(rho_r0=1.0, rho_b0=0.8, nu_r=0.05, nu_b=0.1, sigma=0.003)


def mixed(shape, seed):
    """Both colours everywhere, rough at the grid's scale."""
    rng = np.random.default_rng(seed)
    return (rng.uniform(0.4, 0.6, shape).astype(np.float32), rng.uniform(0.3, 0.5, shape).astype(np.float32),
            rng.uniform(-0.03, 0.03, (3,) + shape).astype(np.float32))


@pytest.mark.parametrize("shape,bc", [((9, 14, 35), (0, 0, 0, 0)), ((33, 5, 31), (1, 1, 1, 1))])
def test_fields_are_the_densities_of_the_step(lb, shape, bc):
    """The total density that the gather pass left for the gradient against rho_r + rho_b of the fields
    of the state that the collision then wrote."""
    import torch
    from paper_1804_08923_gb300 import _abi
    lat = lb.Lattice(shape[::-1], PARAMS, bc=bc)
    lat.init_fields(*mixed(shape, 4))
    for _ in range(2):
        lat.step_gather()
        planes = []
        for z in range(shape[0]):
            buf = torch.empty(lat.halo_bytes(_abi.HALO_PHASE), dtype=torch.uint8, device="cuda")
            lat.halo_pack(_abi.HALO_PHASE, z, buf)
            planes.append(buf)
        lat.step_collide()
        F = lat.fields(("rho_r", "rho_b"))
        torch.cuda.synchronize()
        rho = torch.stack(planes).view(torch.float32).view(shape + (2,))[..., 1]
        assert torch.equal(F["rho_r"] + F["rho_b"], rho)
    lat.close()


@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 1, 1, 1), (1, 3, 0, 0)])
def test_a_uniform_rest_state_keeps_its_densities_from_the_start(lb, bc):
    lat = lb.Lattice((33, 9, 12), PARAMS, bc=bc)
    rng = np.random.default_rng(8)
    for rr, rb in rng.uniform(0.1, 0.9, (12, 2)).astype(np.float32):
        lat.init_uniform(float(rr), float(rb))
        for n in (0, 1, 4):
            lat.step(n)
            F = lat.fields(("rho_r", "rho_b"))
            assert bool((F["rho_r"] == float(rr)).all()) and bool((F["rho_b"] == float(rb)).all()), (n, rr, rb)
    lat.close()
