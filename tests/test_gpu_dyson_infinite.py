"""chi0 with an infinite diagonal entry, in the first pivot block, inside a later
one, and as the last pivot of all: the Dyson step reports a pivot that is not
positive or returns entries that are not numbers, never a finite matrix."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ng", [1, 5, 16, 17, 32, 37, 70])
@pytest.mark.parametrize("where", ["first", "middle", "last"])
def test_infinite_diagonal(ng, where):
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0 as lib
    rng = np.random.default_rng(ng)
    b = rng.standard_normal((ng, 2 * ng)) + 1j * rng.standard_normal((ng, 2 * ng))
    chi = np.stack([-0.02 / ng * (b @ b.conj().T)] * 2)
    v = rng.uniform(0.5, 2.0, ng)
    p = {"first": 0, "middle": ng // 2, "last": ng - 1}[where]
    bad = chi.copy()
    bad[1, p, p] = -np.inf
    stream = torch.cuda.current_stream().cuda_stream
    out = torch.zeros((2, ng, ng), dtype=torch.complex128, device="cuda")
    try:
        lib.invert_eps_noalloc(torch.from_numpy(bad).cuda(), v, out, stream=stream)
        assert not bool(torch.isfinite(torch.view_as_real(out[1])).all())
    except lib.Chi0Error as e:
        assert "ENOTPD" in str(e)
    ok = lib.invert_eps_noalloc(torch.from_numpy(chi).cuda(), v, torch.zeros_like(out), stream=stream)
    ref = np.linalg.inv(np.eye(ng) - v[:, None] * chi[0] * v[None])
    assert np.linalg.norm(ok[1].cpu().numpy() - ref) < 1e-12 * np.linalg.norm(ref)
