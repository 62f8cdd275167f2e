"""Calls that have to work with little device memory: a block of the test's own
leaves the free memory that each one names.  Sizes are some hundred MB, so that
the 2 MB pieces of the device's allocator do not matter.
"""
import contextlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0
    return chi0


@contextlib.contextmanager
def _leave(nbytes):
    """nbytes of device memory left free."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(int(torch.cuda.mem_get_info()[0] - nbytes), dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        torch.cuda.synchronize()
        del fill
        torch.cuda.empty_cache()


def _context(lib, kgrid, L, ng, nocc, nb, nw, qs, fft, seed=1):
    """A mixed-form context on twelve plane waves per state that reach the
    corners of the cube |G_a| <= L."""
    import torch
    rng = np.random.default_rng(seed)
    nk = int(np.prod(kgrid))
    corners = np.array([(L, -L, L), (-L, L, -L), (L, 0, 0), (0, -L, 0), (0, 0, L), (0, 0, 0)])
    box = np.stack(np.meshgrid(*[np.arange(1, L)] * 3, indexing="ij"), -1).reshape(-1, 3)
    ctx = lib.Chi0(a=9.0, kgrid=kgrid, nbands=nb, npw_max=12, fft=fft, ng=ng, q_frac=qs,
                   omega=1j * np.linspace(0.1, 2.0, nw), eta=0.0, precision=lib.CHI0_MIXED_BF16X3,
                   stream=torch.cuda.current_stream().cuda_stream)
    for ik in range(nk):
        g = np.concatenate([corners, box[rng.choice(len(box), 6, replace=False)]]).astype(np.int32)
        c = rng.standard_normal((nb, 12)) + 1j * rng.standard_normal((nb, 12))
        ctx.set_wavefunctions(ik, g, (c / np.linalg.norm(c, axis=1, keepdims=True)).astype(np.complex64))
    e = np.concatenate([rng.uniform(-0.4, 0.0, (nk, nocc)), rng.uniform(0.1, 1.0, (nk, nb - nocc))], 1)
    ctx.set_energies(e, np.broadcast_to((np.arange(nb) < nocc).astype(float), (nk, nb)).copy())
    ctx.synchronize()
    return ctx


def test_batch_keeps_its_first_plan(lib):
    """204,800 transitions of N_G = 250 (390 MB per operand pair): with seven
    pairs of memory left beside states and rho, a batch plans operands of three
    of its four frequencies.  On the scratch sized for that it must not find room
    for the fourth, whose partials would be three times as large."""
    import torch
    nocc, nb, ng, nw = 8, 408, 250, 4
    ctx = _context(lib, (4, 4, 4), 3, ng, nocc, nb, nw, [(0.25, 0.0, 0.0)], (16, 16, 16))
    out = [torch.zeros((nw, ng, ng), dtype=torch.complex128, device="cuda") for _ in range(2)]

    def run():
        batch = lib.Batch([ctx], [0], [out[0]], nstreams=1, chi_out=[out[1]])
        batch.run(torch.cuda.current_stream().cuda_stream)
        batch.synchronize()
        batch.close()
        return [o.cpu().numpy() for o in out]

    ref = run()
    nt = 64 * nocc * (nb - nocc)
    pair = 512 * nt * 4
    with _leave(64 * nb * 12 ** 3 * 8 + nt * ng * 8 + 7 * pair):
        got = run()
    ctx.close()
    for a, b in zip(got, ref):            # the same products, summed in other pieces
        assert np.linalg.norm(a - b) < 1e-6 * np.linalg.norm(b)


def test_operands_of_the_last_q_point_count_as_memory(lib):
    """A metal's transitions with weight differ from q point to q point (here a
    band count per k that differs, 0/1 occupations).  The second q point has more
    of them, so none of the first one's operand pairs is large enough; they hold
    half of the memory, and what they hold has to count, or the eight frequencies
    go in two passes instead of one (seen in the number of kernels launched)."""
    import torch
    rng = np.random.default_rng(5)
    nb, ng, nw = 300, 250, 8
    qs = [(q / 4, 0.0, 0.0) for q in (1, 2)]
    nocc = np.repeat(rng.integers(4, 13, 4), 16)          # by k_x
    ctx = _context(lib, (4, 4, 4), 3, ng, 4, nb, nw, qs, (16, 16, 16))
    e = rng.uniform(0.1, 1.0, (64, nb))
    occ = (np.arange(nb)[None] < nocc[:, None]).astype(float)
    ctx.set_energies(np.where(occ > 0, -e, e), occ)
    rows = [sum(int(nocc[(16 * (kx - iq - 1)) % 64]) * (nb - int(nocc[16 * kx])) * 16 for kx in range(4)) for iq in range(2)]
    order = np.argsort(rows)
    assert rows[order[1]] >= rows[order[0]] + 64
    out = torch.zeros((nw, ng, ng), dtype=torch.complex128, device="cuda")

    def launches(iq):
        ctx.compute_rho(iq)
        before = ctx.get_stats()[3]
        ctx.build_chi0(iq, out)
        ctx.synchronize()
        return ctx.get_stats()[3] - before

    ctx.compute_rho(int(order[0]))                        # states and rho in place
    pair = 512 * rows[order[0]] * 4
    with _leave(17 * pair):
        got = [launches(int(iq)) for iq in order]
    ctx.close()
    assert got[0] == got[1]


# 96,000 states on 12^3 points (1.3 GB) at the first q point and on 15^3 (2.6 GB)
# at the second, whose response set reaches further along x; rho 47 MB and as
# much for a pair of the contraction's operands
NB, NGQ, NWQ = 1500, 61, 8
QQ = [(0.25, 0.0, 0.0), (0.5, 0.0, 0.0)]
STATES, RHO = 64 * NB * 8, 64 * (NB - 1) * NGQ * 8


def _two_q(lib, fft):
    return _context(lib, (4, 4, 4), 4, NGQ, 1, NB, NWQ, QQ, fft, seed=2)


def _rho_and_chi(ctx, iq):
    import torch
    chi = torch.zeros((NWQ, NGQ, NGQ), dtype=torch.complex128, device="cuda")
    ctx.compute_rho(iq)
    rho = ctx.get_rho_rows(np.arange(0, 64 * (NB - 1), 997))
    ctx.build_chi0(iq, chi)
    ctx.synchronize()
    return rho, chi.cpu().numpy()


@pytest.fixture(scope="module")
def ample(lib):
    """The results with all of the memory."""
    ref = []
    for iq in range(2):
        ctx = _two_q(lib, (20, 20, 20))
        ref.append(_rho_and_chi(ctx, iq))
        ctx.close()
    return ref


@pytest.mark.parametrize("fft,room", [
    # what the states of the caller's 20 x 20 grid, 9 planes deep, would take (2.8 GB),
    # and some: those of both q points fit
    ((20, 20, 20), STATES * 20 * 20 * 9 + 3 * RHO),
    # a grid that is just alias free (1404 points): both q points need more than it.
    # The second one's states fit where the first one's operands are given back
    ((13, 12, 12), STATES * 15 ** 3 + 5 * RHO)])
def test_second_q_point_with_larger_states(lib, ample, fft, room):
    ctx = _two_q(lib, fft)
    with _leave(room):
        got = [_rho_and_chi(ctx, iq) for iq in (0, 1, 0)]
    ctx.close()
    for (rho, chi), iq in zip(got, (0, 1, 0)):
        assert np.array_equal(rho, ample[iq][0]), iq     # the same kernels on the same grid
        assert np.linalg.norm(chi - ample[iq][1]) < 1e-6 * np.linalg.norm(chi)


def test_callers_grid_where_the_larger_one_does_not_fit(lib, ample):
    """1.1 GB for the states on the caller's grid, where 15^3 points would take
    2.6: the kernels of the caller's grid, the same sums otherwise rounded (FP32:
    some 15 levels of additions of 6e-8)."""
    ctx = _two_q(lib, (13, 12, 12))
    with _leave(STATES * 1404 + 6 * RHO):
        rho, chi = _rho_and_chi(ctx, 1)
    again = _rho_and_chi(ctx, 1)          # (the plan holds)
    ctx.close()
    assert 0 < np.linalg.norm(rho - ample[1][0]) < 2e-6 * np.linalg.norm(rho)
    assert np.array_equal(rho, again[0])
    assert np.linalg.norm(chi - ample[1][1]) < 5e-6 * np.linalg.norm(chi)


@pytest.mark.parametrize("iqs,states", [((1,), 1404), ((1, 0), 1404 + 12 ** 3), ((0, 1), 12 ** 3 + 1404)])
def test_batch_on_the_callers_grid(lib, ample, iqs, states):
    """The same in a batch, of one system or of two: 2.6 GB for the states of the
    second q point do not fit, its 1.1 GB on the caller's grid do, beside the
    1.3 GB of a first q point of another system."""
    import torch
    ctxs = [_two_q(lib, (13, 12, 12)) for _ in iqs]
    out = [torch.zeros((NWQ, NGQ, NGQ), dtype=torch.complex128, device="cuda") for _ in iqs]
    with _leave(STATES * states + 16 * RHO):
        batch = lib.Batch(ctxs, iqs, [None] * len(iqs), nstreams=1, chi_out=out)
        batch.run(torch.cuda.current_stream().cuda_stream)
        batch.synchronize()
        batch.close()
    for c in ctxs:
        c.close()
    for iq, chi in zip(iqs, out):
        assert np.linalg.norm(chi.cpu().numpy() - ample[iq][1]) < 5e-6 * np.linalg.norm(ample[iq][1])


def test_self_energy_operands_of_fewer_frequencies(lib):
    """N_G = 3000: the operands of W^delta take 72 MB per frequency, 580 MB for the
    eight that go through the split at a time.  With 300 MB left fewer do, and the
    results have the same bits."""
    import torch
    ng, nw, nb = 3000, 8, 6
    ctx = _context(lib, (2, 1, 1), 3, ng, 2, nb, 1, [(0.5, 0.0, 0.0)], (24, 24, 24))
    ctx.compute_rho(0)
    gen = torch.Generator(device="cuda").manual_seed(3)
    eps = torch.randn(nw, ng, ng, dtype=torch.complex128, device="cuda", generator=gen)
    out = torch.zeros((nw, 2, nb, 2, 2), dtype=torch.complex128, device="cuda")
    ctx.synchronize()
    with _leave(300 * MB):
        ctx.build_sigma_i(0, 1, 3, eps, out)
        ctx.synchronize()
    got = out.clone()
    ctx.build_sigma_i(0, 1, 3, eps, out)
    ctx.synchronize()
    ctx.close()
    assert bool((got != 0).any()) and torch.equal(got, out)
