"""The Dyson step at the sizes between which the number of update blocks changes:
alone (N_G = 900 and 1009, below and above), and in the pipeline with the
contraction, where matrices as long as the pivot chain also go in two groups
(N_G = 700 and 760).  Every entry is the same sum whatever the blocks, so the
pipeline gives the bits of the separate calls; against numpy 1e-12 (condition
numbers below 10, sums of 1000 terms at 1e-16)."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("ng,nw", [(900, 2), (1009, 3)])
def test_alone(lib, ng, nw):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(ng)
    b = torch.randn(nw, ng, 2 * ng, dtype=torch.complex128, device="cuda", generator=gen)
    chi = -(b @ b.mH) * (0.5 / ng)
    v = np.linspace(0.5, 2.0, ng)
    out = lib.invert_eps_noalloc(chi, v, torch.empty_like(chi), stream=torch.cuda.current_stream().cuda_stream)
    for c, o in zip(chi.cpu().numpy(), out.cpu().numpy()):
        ref = np.linalg.inv(np.eye(ng) - v[:, None] * c * v[None])
        assert np.linalg.norm(o - ref) < 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("ng,freqs,eta", [(700, (0.1j, 0.9j, 3.0j), 0.0), (760, (0.1j, 0.9j), 0.0),
                                          (760, (0.1j, 0.9j, 3.0j), 0.0), (760, (0.1j, 0.3, 0.5, 0.8, 2.0j), 0.004),
                                          (550, (0.2, 0.4, 0.6), 0.004)])
def test_in_the_pipeline(lib, ng, freqs, eta):
    import torch
    s = make_system(cfg_tiny(seed=31, kgrid=(2, 1, 1), q_frac=((0.5, 0.0, 0.0),), fft=(24, 24, 24), ng=ng, n_occ=3,
                             n_bands=9, npw_target=60, a=8.0, freqs=freqs, eta=eta, coef_dtype="c64"))
    ctx = lib.Chi0.for_system(s, precision=1, stream=torch.cuda.current_stream().cuda_stream)
    ctx.load_system(s)
    ctx.compute_rho(0)
    one, two = (torch.zeros((len(freqs), ng, ng), dtype=torch.complex128, device="cuda") for _ in range(2))
    chi = torch.zeros_like(one)
    ctx.build_invert(0, one, chi)
    ctx.build_chi0(0, None)
    ctx.invert_eps(0, two)
    ctx.synchronize()
    ctx.close()
    assert bool((chi != 0).any()) and torch.equal(one, two)
