"""One context over q points whose grids differ: the states at q = (1/4, 0, 0)
are on 12^3 points, at q = (1/2, 0, 0) on 15^3 (a response set that reaches one
vector further along x).  The loop gives each q point the bits of a context of
its own; a call that fails on the way (no memory, a caller's grid that aliases
at one of them) leaves nothing that a later call could take for a plan or a
result, and the same call works once the cause is gone.
"""
import numpy as np
import pytest

import oracle as O
from synth import cfg_tiny, make_system

pytestmark = pytest.mark.gpu

QS = ((0.25, 0.0, 0.0), (0.5, 0.0, 0.0))


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0
    return chi0


def _system(prec, fft):
    s = make_system(cfg_tiny(seed=11, kgrid=(4, 1, 1), q_frac=QS, fft=fft, ng=61, n_occ=3, n_bands=9,
                             npw_target=170, freqs=(0.2j, 1.1j), eta=0.0, coef_dtype="c64" if prec else "c128"))
    assert np.abs(s.gvec).max() == 4      # the grids that the text above names
    return s


def _context(lib, s, prec):
    import torch
    ctx = lib.Chi0.for_system(s, precision=prec, stream=torch.cuda.current_stream().cuda_stream)
    ctx.load_system(s)
    return ctx


def _results(ctx, s, iq):
    ctx.compute_rho(iq)
    rho = ctx.get_rho()
    chi = np.zeros((s.freqs.size, s.ng, s.ng), np.complex128)
    inv = np.zeros_like(chi)
    ctx.build_invert(iq, inv, chi)
    return rho, chi, inv


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.fixture(scope="module", params=[0, 1])
def case(lib, request):
    """(precision, system, results of each q point in a context of its own)"""
    prec = request.param
    s = _system(prec, (13, 12, 12))
    ref = []
    for iq in range(2):
        ctx = _context(lib, s, prec)
        ref.append(_results(ctx, s, iq))
        rho = O.rho_transitions(s, iq, O.response_gvectors(s.spec.kgrid, QS[iq], s.ng), ctx.get_transitions())
        ctx.close()
        # FP64: some 15 levels of additions of 1.1e-16; FP32: the same at 6e-8
        assert np.linalg.norm(ref[iq][0] - rho) < (2e-6 if prec else 1e-13) * np.linalg.norm(rho)
    return prec, s, ref


def test_q_loop(lib, case):
    prec, s, ref = case
    ctx = _context(lib, s, prec)
    for iq in (0, 1, 1, 0, 1, 0, 0):
        assert _same(_results(ctx, s, iq), ref[iq]), iq
    ctx.close()


@pytest.mark.parametrize("first", [0, 1])
def test_retry_after_a_failed_allocation(lib, case, monkeypatch, first):
    prec, s, ref = case
    ctx = _context(lib, s, prec)
    if first == 0:                        # the states have to grow for the second q point
        assert _same(_results(ctx, s, 0), ref[0])
    monkeypatch.setenv("CHI0_FAULT", "alloc")
    with pytest.raises(lib.Chi0Error, match="ENOMEM"):
        ctx.compute_rho(1)
    with pytest.raises(lib.Chi0Error, match="ENOMEM"):
        ctx.compute_rho(1)
    with pytest.raises(lib.Chi0Error, match="ESTATE"):
        ctx.get_rho()
    monkeypatch.delenv("CHI0_FAULT")
    for iq in (1, 0, 1):
        assert _same(_results(ctx, s, iq), ref[iq]), iq
    ctx.close()


def test_q_point_that_the_grid_cannot_take(lib, case):
    import torch
    prec, _, ref = case
    s = _system(prec, (12, 12, 12))       # alias free at the first q point only
    ctx = _context(lib, s, prec)
    assert _same(_results(ctx, s, 0), ref[0])
    eps = torch.zeros((s.freqs.size, s.ng, s.ng), dtype=torch.complex128, device="cuda")
    out = torch.zeros((s.freqs.size, 4, 9, 2, 2), dtype=torch.complex128, device="cuda")
    for _ in range(2):
        with pytest.raises(lib.Chi0Error, match="EINVAL"):
            ctx.compute_rho(1)
        for iq in range(2):               # neither q point has a rho now
            with pytest.raises(lib.Chi0Error, match="ESTATE"):
                ctx.build_chi0(iq, eps)
            with pytest.raises(lib.Chi0Error, match="ESTATE"):
                ctx.build_sigma_i(iq, 2, 4, eps, out)
        assert _same(_results(ctx, s, 0), ref[0])
    ctx.close()
