"""Fragment labelling where runs of jet nodes meet the ends of rows, of a warp's 32 nodes and of the
lattice: random fields of several densities on extents around those lengths, periodic and walled,
both neighbourhoods, against the oracle's flood fill (exact lists); and more fragments than the
binding's first guess of their number."""
import numpy as np
import pytest

from test_gpu_fragments import both, lb, same  # noqa: F401  (lb is the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 5, 33), (9, 7, 1), (65, 3, 2), (3, 1, 70), (2, 2, 31), (3, 4, 32), (5, 6, 64), (1, 9, 40)])
@pytest.mark.parametrize("bc", [(0, 0), (0, 0, 1, 0), (0, 0, 1, 1)])
def test_runs_at_every_edge(lb, shape, bc):  # noqa: F811
    for seed, fill in enumerate((0.15, 0.4, 0.75)):
        jet = np.random.default_rng(seed).random(shape) < fill
        gpu, ref = both(lb, jet, bc=bc)
        for conn in (6, 26):
            same(gpu.fragments(conn), ref.fragments(conn))


def test_more_fragments_than_the_first_guess(lb):  # noqa: F811
    jet = np.zeros((34, 34, 34), bool)
    jet[::2, ::2, ::2] = True
    gpu, ref = both(lb, jet)
    g = gpu.fragments(6)
    same(g, ref.fragments(6))
    assert len(g["roots"]) == 17 ** 3
