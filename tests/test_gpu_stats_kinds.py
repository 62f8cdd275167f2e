"""Stage times of many unread passes whose instances of a stage differ: with the
extrapolar correction a pass computes rho of the transitions (long) and the
diagonal densities (short), both in the rho stage.  The mean over 2000 passes,
most of them sampled, must be that of 200 passes that are all timed.  Bound: the
sampled calls stand for one window of 16 each, so their number is right to 1%,
and the kernels' times spread by some 10%; one kind standing for both would
double the sum.
"""
import pytest

from synth import cfg_tiny, make_system

pytestmark = pytest.mark.gpu


def test_rho_stage_with_diagonal_densities():
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0 as lib
    s = make_system(cfg_tiny(seed=6, kgrid=(4, 4, 2), q_frac=((0.25, 0.0, 0.0),), fft=(24, 24, 24), ng=60, n_occ=4,
                             n_bands=90, npw_target=140, a=8.0, freqs=(0.2j,), eta=0.0, coef_dtype="c64"))
    ctx = lib.Chi0.for_system(s, precision=1, stream=torch.cuda.current_stream().cuda_stream)
    ctx.load_system(s)
    ctx.set_bg_terminator(1.5)
    out = torch.zeros((1, s.ng, s.ng), dtype=torch.complex128, device="cuda")

    def passes(n):
        for i in range(n):
            ctx.compute_rho(0)
            ctx.build_chi0(0, out)
            if i % 100 == 99:
                ctx.synchronize()
        return ctx.get_stats()[0]["rho"] / n

    passes(50)
    first, many = passes(200), passes(2000)
    ctx.close()
    assert abs(many - first) < 0.25 * first, (first, many)


@pytest.mark.parametrize("n", [15, 23, 31, 40, 90])
def test_calls_of_many_instances(n):
    """A call of some 25 stages: the calls beyond the first twenty or so are sampled,
    and the mean over n calls must be that of five, however few of them were
    (bound as above)."""
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0 as lib
    s = make_system(cfg_tiny(seed=7, kgrid=(4, 4, 2), q_frac=((0.25, 0.0, 0.0),), fft=(24, 24, 24), ng=120, n_occ=4,
                             n_bands=60, npw_target=140, a=8.0, freqs=tuple(0.1j * (i + 1) for i in range(64)), eta=0.0,
                             coef_dtype="c64"))
    ctx = lib.Chi0.for_system(s, precision=1, stream=torch.cuda.current_stream().cuda_stream)
    ctx.load_system(s)
    ctx.compute_rho(0)

    def calls(k):
        for _ in range(k):
            ctx.build_chi0(0, None)
        ctx.synchronize()
        return {name: ms / k for name, ms in ctx.get_stats()[0].items()}

    calls(5)
    first, many = calls(5), calls(n)
    ctx.close()
    for name in ("weights", "contract", "reduce"):
        assert abs(many[name] - first[name]) < 0.25 * first[name], (name, first, many)
