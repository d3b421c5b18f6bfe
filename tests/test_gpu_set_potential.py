"""gpe_create and gpe_set_problem take V through a check and a conversion on the
device: host and device sources, one off an 8-byte boundary's neighbour, extremes
of both signs (signed zeros among them), non-finite values at the first, a middle
and the last point, which are refused and leave the context as it was."""
import numpy as np
import pytest

from oracle import gpe_oracle as O
from paper_1611_02045_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G(built_lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_02045_gb300 import gpe
    return gpe


def _potentials(n, L):
    h = I.harmonic(n, L)
    z = h.copy()
    z.flat[0], z.flat[-1] = -0.0, 0.0
    return {"positive": h, "negative": -h - 3.0, "both": h - 5.0, "zeros": z * 0.0, "signed zeros": z}


@pytest.mark.parametrize("n", [(8, 8), (64, 16), (16, 8, 32), (256, 256)])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_potential_sources(G, n, prec):
    L = tuple(5.0 for _ in n)
    dt, tol = (torch.complex128, 1e-12) if prec == 0 else (torch.complex64, 2e-5)
    phi = torch.from_numpy(I.random_field(1, n, L)).to("cuda", dt)
    out = torch.empty_like(phi)
    ph = phi.cpu().numpy().astype(complex)
    with G.Context(n, L, 3.0, 0.4, np.zeros(I.shape_of(n)), prec=prec) as ctx:
        for name, V in _potentials(n, L).items():
            pad = torch.zeros(V.size + 1, dtype=torch.float64, device="cuda")
            pad[1:] = torch.from_numpy(V.ravel()).cuda()
            want = O.apply_H(O.Problem(n, L, 3.0, 0.4, V), ph, ph)
            for src in (V, torch.from_numpy(V.copy()), torch.from_numpy(V.copy()).cuda(), pad[1:]):
                ctx.set_problem(src)
                if torch.is_tensor(src):
                    src.fill_(1e30)  # the caller's buffer is its own again
                ctx.apply_H(phi, phi, out)
                assert np.max(np.abs(out.cpu().numpy() - want)) <= tol * np.max(np.abs(want)), name
                pad[1:] = torch.from_numpy(V.ravel()).cuda()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("where", [0, 1, -1])
def test_non_finite_potential_is_refused(G, bad, where):
    n, L = (64, 32), (4.0, 4.0)
    V = I.harmonic(n, L)
    Vb = V.copy()
    at = {0: 0, 1: V.size // 2 + 1, -1: V.size - 1}[where]
    Vb.flat[at] = bad
    for src in (Vb, torch.from_numpy(Vb).cuda()):
        with pytest.raises(G.GpeError) as e:
            G.Context(n, L, 1.0, 0.0, src)
        assert e.value.status == G.GPE_ERR_ARG
    phi = torch.from_numpy(I.random_field(1, n, L)).cuda()
    a, b = torch.empty_like(phi), torch.empty_like(phi)
    with G.Context(n, L, 9.0, 0.1, V) as ctx:
        ctx.apply_H(phi, phi, a)
        mu = ctx.thomas_fermi(b)
        for src in (Vb, torch.from_numpy(Vb).cuda()):
            with pytest.raises(G.GpeError) as e:
                ctx.set_problem(src, 7.0, 0.2)
            assert e.value.status == G.GPE_ERR_ARG
        ctx.apply_H(phi, phi, b)
        assert torch.equal(a, b) and ctx.thomas_fermi(b) == mu
