"""chi0 and eps~^-1 of a metal, where many transitions of the (k, n, m) block
carry no weight (f_m - f_n <= 0) and are left out of the contraction: both
forms, imaginary- and real-axis frequencies together, with the double grid and
with pole groups too small for the grouped contraction, against the oracle
(which drops nothing).  Tolerances as elsewhere: 1e-10 (FP64), 1e-5 (mixed).
"""
import dataclasses

import numpy as np
import pytest

import oracle as O
from synth import cfg_tiny, make_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0
    return chi0


def _metal(dtype, ng):
    spec = cfg_tiny(seed=17, kgrid=(3, 2, 1), q_frac=((1 / 3, 0.5, 0.0),), fft=(18, 18, 18), ng=ng, n_occ=0,
                    n_bands=13, npw_target=50, a=8.0, freqs=(0.05j, 0.6j, 0.4 + 0j), eta=0.05, coef_dtype=dtype)
    return make_system(dataclasses.replace(spec, occ_ev=(-10.0, 30.0), emp_ev=(-10.0, 30.0), kT_ev=0.3,
                                           n_electrons=8))


@pytest.mark.parametrize("prec,dtype,tol", [(0, "c128", 1e-10), (1, "c64", 1e-5)])
@pytest.mark.parametrize("option,ng", [("plain", 33), ("plain", 70), ("dense", 33), ("groups", 33)])
def test_metal_rows_vs_oracle(lib, prec, dtype, tol, option, ng):
    import torch
    s = _metal(dtype, ng)
    G = O.response_gvectors(s.spec.kgrid, s.q_frac[0], s.ng)
    ctx = lib.Chi0.for_system(s, precision=prec, occ_drop_tol=1e-12,
                              stream=torch.cuda.current_stream().cuda_stream)
    ctx.load_system(s)
    if option == "dense":
        rng = np.random.default_rng(2)
        dense = s.eps[:, None, :] + 0.01 * rng.uniform(-1.0, 1.0, (s.nk, 3, s.nb))
        ctx.set_double_grid(dense)
        ref = O.chi0_double_grid(s, 0, G, s.freqs, s.eta, dense)
    elif option == "groups":
        ctx.set_pole_grouping(1e-3)
        ref = O.chi0_grouped(s, 0, G, s.freqs, s.eta, 1e-3, occ_tol=1e-12)   # the groups of the same rows
    else:
        ref = O.chi0_tr(s, 0, G, s.freqs, s.eta)
    ctx.compute_rho(0)
    t = ctx.get_transitions()
    kq = O.kpair_map(s.spec.kgrid, s.q_frac[0])[0]
    df = s.occ[kq[t[:, 0]], t[:, 2]] - s.occ[t[:, 0], t[:, 1]]
    assert (df > 1e-12).mean() < 7 / 8    # rows are left out
    chi = np.zeros((s.freqs.size, s.ng, s.ng), np.complex128)
    inv = np.zeros_like(chi)
    ctx.build_invert(0, inv, chi)
    ctx.close()
    qg = O.qg_norms(s.spec.a, s.q_frac[0], G)
    for w in range(s.freqs.size):
        assert np.linalg.norm(chi[w] - ref[w]) < tol * np.linalg.norm(ref[w])
        e = O.eps_inv_gauss_jordan(ref[w], qg)
        assert np.linalg.norm(inv[w] - e) < tol * np.linalg.norm(e)
