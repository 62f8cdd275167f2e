"""Two threads, each with a context and a stream of its own, whose launches of the
same kernels take different amounts of shared memory (response sets of 7 and of
200 vectors on the same grid, 30 points or the caller's 44): every call succeeds,
and each thread gets the bits that it gets alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fft,calls", [((32, 32, 32), 3000), ((44, 44, 44), 1000)])
def test_contexts_with_different_shared_memory(fft, calls):
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0 as lib

    # a sphere of few vectors that needs column transforms of 30 points, or more than there are
    far = 12 if fft[0] == 32 else 18
    gvec = np.array([(far, 0, 0), (-far, 0, 0), (0, 1, 0), (0, 0, -1), (0, 0, 0), (1, -1, 1)], np.int32)

    def context(ng, stream):
        rng = np.random.default_rng(ng)
        ctx = lib.Chi0(a=9.0, kgrid=(2, 1, 1), nbands=4, npw_max=len(gvec), fft=fft, ng=ng, q_frac=[(0.5, 0, 0)],
                       omega=[0.3j], eta=0.0, precision=lib.CHI0_MIXED_BF16X3, stream=stream.cuda_stream)
        for ik in range(2):
            c = rng.standard_normal((4, len(gvec))) + 1j * rng.standard_normal((4, len(gvec)))
            ctx.set_wavefunctions(ik, gvec, c.astype(np.complex64))
        e = np.stack([np.array([-0.3, -0.1, 0.2, 0.5])] * 2)
        ctx.set_energies(e, (e < 0).astype(float))
        ctx.compute_rho(0)
        return ctx, ctx.get_rho()

    failed = []

    def run(ctx, want):
        try:
            for _ in range(calls):
                ctx.compute_rho(0)
            if not np.array_equal(ctx.get_rho(), want):
                failed.append("other bits")
        except lib.Chi0Error as e:
            failed.append(str(e))

    streams = [torch.cuda.Stream() for _ in range(2)]
    parts = [context(ng, s) for ng, s in zip((7, 200), streams)]
    threads = [threading.Thread(target=run, args=p) for p in parts]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ctx, _ in parts:
        ctx.close()
    assert not failed, failed
