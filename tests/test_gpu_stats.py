"""Stage times after many unread passes: beyond 512 instances of a stage every
16th is timed and stands for its neighbours, so the sum must stay that of all
passes.  Loose bounds (a factor of three either way on the mean of the passes
that are all timed): they tell a sum that lost or repeated instances (1.2 and
19 times) from one that has them all.
"""
import pytest

from synth import cfg_tiny, make_system

pytestmark = pytest.mark.gpu


def test_stage_times_of_many_passes():
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0 as lib
    s = make_system(cfg_tiny(seed=5, freqs=(0.1j,), eta=0.0))
    ctx = lib.Chi0.for_system(s, stream=torch.cuda.current_stream().cuda_stream)
    ctx.load_system(s)
    for _ in range(50):
        ctx.compute_rho(0)
    ctx.get_stats()                      # warm-up
    for _ in range(200):
        ctx.compute_rho(0)
    first = ctx.get_stats()[0]["rho"] / 200
    n = 6000
    for i in range(n):
        ctx.compute_rho(0)
        if i % 500 == 499:
            ctx.synchronize()            # finished pairs are folded and used again
    many = ctx.get_stats()[0]["rho"] / n
    assert first / 3 < many < 3 * first, (first, many)
    assert ctx.get_stats()[0]["rho"] == 0.0
    ctx.close()
