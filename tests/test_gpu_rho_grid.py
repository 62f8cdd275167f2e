"""rho at every size of the column transforms (the smallest alias-free grid is
chosen by the library: 2 L + max|G - G0| + 1 points, rounded up to 8, 10, 12,
15, 16, 18, 20, 24, 30, 32 or 36) and where none fits (the caller's grid).

Two k points with an umklapp pair, twelve plane waves per state that reach the
corners of the cube |G_a| <= L, odd and even numbers of bands on both sides;
against the oracle's direct convolution.  Tolerances (relative Frobenius): FP64
1e-13, some 15 levels of additions of 1.1e-16 each; FP32 2e-6, the same levels
at 6e-8 and the rounding of the states.
"""
import dataclasses

import numpy as np
import pytest

import oracle as O
from synth import cfg_tiny, make_system

pytestmark = pytest.mark.gpu

# (grid the plan takes, 0 = the caller's; L; N_G)
SIZES = [(8, 2, 7), (10, 3, 7), (12, 4, 7), (15, 6, 7), (16, 6, 19), (18, 7, 7), (20, 8, 19), (24, 10, 19)]
FP32_SIZES = SIZES + [(30, 13, 7), (32, 14, 7), (36, 13, 700), (0, 14, 300)]
FP64_SIZES = SIZES + [(30, 10, 300), (0, 11, 40)]


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0
    return chi0


def _system(L, ng, n_occ, n_bands, dtype, seed):
    q = (0.5, 0.0, 0.0)
    G = O.response_gvectors((2, 1, 1), q, ng)
    need = 2 * L + int(np.abs(G).max()) + 2
    s = make_system(cfg_tiny(seed=seed, kgrid=(2, 1, 1), q_frac=(q,), fft=(need, need + 1, need + 3), ng=ng,
                             n_occ=n_occ, n_bands=n_bands, npw_target=30, freqs=(0.3j,), eta=0.0, coef_dtype=dtype))
    rng = np.random.default_rng(seed)
    corners = np.array([(L, -L, L), (-L, L, -L), (L, 0, 0), (0, -L, 0), (0, 0, L), (0, 0, 0)])
    gvec = np.zeros((2, 12, 3), np.int32)
    for ik in range(2):
        more = rng.integers(-L, L + 1, (40, 3))
        g = np.unique(np.concatenate([corners, more]), axis=0)
        keep = [tuple(v) in {tuple(c) for c in corners} for v in g]
        rest = np.nonzero(~np.array(keep))[0][:6]
        gvec[ik] = np.concatenate([corners, g[rest]])
    c = rng.standard_normal((2, n_bands, 12)) + 1j * rng.standard_normal((2, n_bands, 12))
    c /= np.linalg.norm(c, axis=2, keepdims=True)
    return need, dataclasses.replace(s, npw=np.full(2, 12, np.int32), gvec=gvec,
                                     coef=c.astype(np.complex64 if dtype == "c64" else np.complex128))


def _points(L, G):
    """Points per axis that the plan asks for."""
    h = int(np.abs(G).max()) + 1
    return max(2 * L + h + 1, 2 * h + 1)


@pytest.mark.parametrize("prec,size", [(0, v) for v in FP64_SIZES] + [(1, v) for v in FP32_SIZES])
@pytest.mark.parametrize("bands", [(1, 4), (3, 8), (6, 9)])
def test_rho_on_every_grid(lib, prec, size, bands):
    import torch
    n, L, ng = size
    need, s = _system(L, ng, bands[0], bands[1], "c64" if prec else "c128", 100 + L)
    G = O.response_gvectors(s.spec.kgrid, s.q_frac[0], ng)
    taken = [v for v in (8, 10, 12, 15, 16, 18, 20, 24, 30, 32, 36) if v >= _points(L, G)][0]
    room = (taken * (2 * L + 1) ** 2 + taken * (2 * L + 1)) * (8 if prec else 16) <= 227 * 1024
    assert (taken if room else 0) == n    # the case covers the size that it names
    ctx = lib.Chi0.for_system(s, precision=prec, stream=torch.cuda.current_stream().cuda_stream)
    ctx.load_system(s)
    ctx.compute_rho(0)
    got = ctx.get_rho()
    ref = O.rho_transitions(s, 0, G, ctx.get_transitions())
    ctx.close()
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err < (2e-6 if prec else 1e-13), err
