"""Failures inside a call of several steps, made on the host: launches that the runtime refuses, and the
error flag as a bounded wait that ran out leaves it."""
import ctypes as C
import os

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

LB_ECUDA, LB_ETIMEOUT = 3, 5
GRID = (96, 64, 96)  # large enough for the advance


@pytest.fixture(scope="module")
def lb(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import native
    import paper_1804_08923_gb300 as lbm
    from paper_1804_08923_gb300 import _abi
    path = str(tmp_path_factory.mktemp("faults") / "liblbcm_faults.so")
    lbm.faults = native.wrapped(os.path.join(os.path.dirname(__file__), "launch_faults.cu"), path,
                                {"STEP": "launch_step", "ADVANCE": "launch_advance"}).launch_faults
    kept, _abi._lib = _abi._lib, None
    _abi.library(path)
    yield lbm
    _abi._lib = kept
    del lbm.faults


def lattice(lb, bc=(0, 0), **params):
    p = dict(rho_r0=1.0, rho_b0=0.5, nu_r=0.02, nu_b=0.05, sigma=0.003, u_in=0.05, d_in=20.0, **params)
    lat = lb.Lattice(GRID, p, bc=bc)
    lat.init_fields(*workloads.random_two_phase_fields(GRID[::-1], 3, 1.0, 0.5, u_amp=0.03))
    return lat


READERS = {
    "fields": lambda lat: lat.fields(("phi",), device=False),
    "populations": lambda lat: lat.populations(device=False),
    "history": lambda lat: lat.history(),
    "save": lambda lat: lat.save(),
    "fragments": lambda lat: lat.fragments(),
    "halo": lambda lat: lat.halo_pack(0, 1, np.empty(lat.halo_bytes(0), np.uint8)),
    "mass": lambda lat: lat.mass(),
    "mass_planes": lambda lat: lat.mass_planes(0, 2),
    "adjoint": lambda lat: lat.adjoint(2),
}


@pytest.mark.parametrize("read", READERS)
def test_a_wait_that_ran_out_is_reported_by_the_call_that_reads_the_state(lb, read):
    lat = lattice(lb)
    lb.faults(0, 0, 1)
    lat.step(3)
    lb.faults(0, 0, 0)
    with pytest.raises(lb.LBError) as e:
        READERS[read](lat)
    assert e.value.status == LB_ETIMEOUT
    READERS[read](lat)  # once
    lat.close()


def test_a_new_state_is_not_blamed_for_the_last_one(lb):
    lat = lattice(lb)
    blob = lat.save()
    for renew in (lambda: lat.load(blob), lambda: lat.init_uniform(0.3, 0.4)):
        lb.faults(0, 0, 1)
        lat.step(3)
        lb.faults(0, 0, 0)
        renew()
        lat.mass()
    lat.close()


def test_the_advance_s_wait_gives_up(lb):
    """2^14 tries of a barrier wait that cannot succeed: well under a second, and the context steps on."""
    lat, ref = lattice(lb), lattice(lb)
    status, ms = lat.selftest_advance_wait()
    assert status == LB_ETIMEOUT
    assert 1.0 <= ms <= 1000.0, ms
    lat.step(4)
    ref.step(4)
    assert np.array_equal(lat.populations(device=False), ref.populations(device=False))
    lat.close()
    ref.close()


def test_a_refused_launch_leaves_a_whole_state(lb):
    """The k-th launch of a call of six steps fails.  What the context holds then, populations and
    outflow plane, is the state of the step it names; where that is not to be had, it holds none."""
    for bc in ((0, 0), (2, 3)):
        lat, ref = lattice(lb, bc), lattice(lb, bc)
        for k in range(1, 6):
            blob, t = lat.save(), lat.step_count
            lb.faults(0, k, 0)
            with pytest.raises(lb.LBError) as e:
                lat.step(6)
            lb.faults(0, 0, 0)
            assert e.value.status == LB_ECUDA
            assert lat.step_count == t + k  # the first launch of the six is the gather pass
            ref.load(blob)
            for _ in range(k):
                ref.step(1)
            assert np.array_equal(lat.populations(device=False), ref.populations(device=False))
            assert np.array_equal(lat.history(), ref.history())
        blob = lat.save()
        for n, call in ((4, 1), (2, 2), (3, 2)):  # the gather pass of four steps, the collision pass of two and three
            lat.load(blob)
            lb.faults(call, 0, 0)
            with pytest.raises(lb.LBError) as e:
                lat.step(n)
            lb.faults(0, 0, 0)
            assert e.value.status == LB_ECUDA
            if call == 1 or bc[1] != 3:
                assert lat.save() == blob
            else:
                with pytest.raises(lb.LBError):
                    lat.populations()
        lat.close()
        ref.close()


@pytest.mark.parametrize("grid,fail,done", [((24, 16, 20), (3, 0), 2), (GRID, (0, 2), 0), (GRID, (2, 0), 0)])
def test_a_refused_launch_in_an_adjoint_leaves_a_whole_state(lb, grid, fail, done):
    p = dict(rho_r0=1.0, rho_b0=0.5, nu_r=0.02, nu_b=0.05, sigma=0.003, u_in=0.05, d_in=8.0)
    lat, ref = (lb.Lattice(grid, p, bc=(2, 3)) for _ in range(2))
    for l in (lat, ref):
        l.init_fields(*workloads.random_two_phase_fields(grid[::-1], 3, 1.0, 0.5, u_amp=0.03))
    lb.faults(*fail, 0)
    with pytest.raises(lb.LBError) as e:
        lat.adjoint(4, "area", (1e-3,), checkpoint=4)
    lb.faults(0, 0, 0)
    assert e.value.status == LB_ECUDA
    ref.step(done)
    assert lat.step_count == done
    assert np.array_equal(lat.populations(device=False), ref.populations(device=False))
    assert np.array_equal(lat.history(), ref.history())
    lat.close()
    ref.close()
