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


def test_the_automatic_schedule_leaves_the_memory_to_others(lb):
    """200 steps recorded take 14.7 KB a node, with checkpoints every 15 steps 5.7.  After the call all but
    twice the latter can be allocated again; the results are those of a schedule that is named, and the
    next call finds its records."""
    import torch
    T, k, nseg = 200, 15, 14
    lat, ref = lattice(lb), lattice(lb)
    start = lat.save()
    J, _ = ref.adjoint(T, checkpoint=T)
    state = ref.adjoint_state(device=True).clone()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    checkpoints = lat.nodes * (nseg * 216 + 2 * 216 + 2 * k * 72) * (1 + 4.0 / GRID[2])  # and the outflow plane's share
    kept = 2 * checkpoints + lat.nodes * 200 + (256 << 20)
    assert lat.nodes * T * 72 > kept + (1 << 30)
    for _ in range(2):
        lat.load(start)
        assert lat.adjoint(T)[0] == J
        assert torch.equal(lat.adjoint_state(device=True), state)
        torch.cuda.empty_cache()
        others = torch.empty(int(before - kept), dtype=torch.uint8, device="cuda")
        del others
        torch.cuda.empty_cache()
    # a later call that needs less gives back what it does not need
    lat.adjoint(T, checkpoint=T)
    lat.adjoint(3)
    torch.cuda.empty_cache()
    assert before - torch.cuda.mem_get_info()[0] <= lat.nodes * (3 * 72 * 4 + 2 * 216 * 4 + 200) + (256 << 20)
    lat.close()
    ref.close()


def test_a_number_of_steps_beyond_any_memory_is_refused(lb):
    lat = lattice(lb, (16, 8, 10))
    for T, k in ((1 << 50, 1 << 50), (1 << 62, 0), (1 << 62, 1)):
        with pytest.raises(lb.LBError) as e:
            lat.adjoint(T, checkpoint=k)
        assert e.value.status == 2  # LB_ENOMEM
    assert np.isfinite(lat.adjoint(2)[0])
    lat.close()


def run(lat, T, objective, args, checkpoint):
    J, g = lat.adjoint(T, objective, args, checkpoint)
    return J, g, lat.adjoint_state(device=True).clone()


@pytest.mark.parametrize("grid,bc", [(GRID, (2, 3)), (GRID, (0, 0)), ((125, 99, 95), (2, 3, 1, 1)), ((70, 66, 400), (1, 1, 1, 1))])
def test_segments_of_recorded_advances(lb, grid, bc):
    """Twelve steps in one recorded segment against six of two and four of three, recomputed by
    advances on the second stream into two alternating sets, and against single steps, which are
    recorded by the two passes: the same bits."""
    import torch
    T = 12
    want = None
    for checkpoint in (T, 2, 3, 5, 1):
        lat = lattice(lb, grid, bc, g=(1e-6, 0.0, 1e-5))
        got = run(lat, T, "area", (1e-3,), checkpoint)
        end = lat.populations().clone()
        if want is None:
            want, want_end = got, end
        assert got[0] == want[0] and np.array_equal(got[1], want[1]), checkpoint
        assert torch.equal(got[2], want[2]) and torch.equal(end, want_end), checkpoint
        lat.close()
