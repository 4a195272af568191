"""lb_step(n) against n single steps, as in test_gpu_advance.py, on lattices where the advance's 16 x 30
tile is the one chosen: whole tiles, one node over and one short, every boundary."""
import pytest

from test_gpu_advance import C, I, P, S, lb, pair, same  # noqa: F401 (lb is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,bc", [((112, 90, 100), (S, S, S, P)), ((177, 148, 60), (P, P, P, P)),
                                     ((145, 119, 80), (I, C, P, P)), ((111, 89, 110), (I, C, S, S))])
def test_several_steps_equal_single_steps_in_tall_tiles(lb, grid, bc):  # noqa: F811
    params = dict(rho_r0=1.0, rho_b0=0.4, nu_r=0.01, nu_b=0.03, sigma=0.004, g=(1e-6, -2e-6, 1e-5), u_in=0.05,
                  d_in=0.4 * min(grid[:2]), noise_amp=0.02, seed=9, fourier=(0.05, 0.02, -0.03))
    a, b = pair(lb, grid, params, bc, 3)
    l0 = a.kernel_launches
    a.step(4)
    assert a.kernel_launches - l0 == 5 + (bc[0] != P), "the advance was not taken"
    for _ in range(4):
        b.step(1)
    same(a, b)
