"""chi0_get_response_gvectors at sizes and q points where the ball that the search
is limited to is cut by the box of candidates or sits off-centre, against the
same order (|q + G|^2 exactly, ties by x, y, z) over every vector of the box."""
import math

import numpy as np
import pytest


@pytest.fixture(scope="module")
def binding():
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0
    return chi0


def _all_sorted(kgrid, q, ng):
    scale = math.lcm(*kgrid)
    lq = np.array([round(q[d] * kgrid[d]) * (scale // kgrid[d]) for d in range(3)])
    m = math.ceil((3.0 * ng / (4.0 * math.pi)) ** (1.0 / 3.0)) + 3
    g = np.stack(np.meshgrid(*[np.arange(-m, m + 1)] * 3, indexing="ij"), -1).reshape(-1, 3)
    n2 = ((lq + scale * g) ** 2).sum(1)
    return g[np.lexsort((g[:, 2], g[:, 1], g[:, 0], n2))[:ng]]


@pytest.mark.parametrize("ng", [1, 2, 3, 7, 8, 20, 33, 57, 250, 1000, 4096])
@pytest.mark.parametrize("kgrid,q", [((1, 1, 1), (0, 0, 0)), ((4, 4, 4), (0.75, 0.75, 0.75)), ((2, 3, 5), (0.5, 2 / 3, 0.8)),
                                     ((4, 2, 1), (-0.75, 0.5, 0)), ((2, 2, 2), (3.5, -4.0, 0.5)), ((1, 1, 2), (40.0, 0, 0.5))])
def test_every_vector_of_the_box(binding, kgrid, q, ng):
    c = binding.Chi0(a=9.0, kgrid=kgrid, nbands=2, npw_max=1, fft=(8, 8, 8), ng=ng, q_frac=[q], omega=[1j], eta=0.0)
    got = c.get_response_gvectors(0)
    c.close()
    assert np.array_equal(got, _all_sorted(kgrid, q, ng))
