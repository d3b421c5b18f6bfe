"""H phi on one square complex64 field of 32 .. 128 points per side (one cluster)
against the passes (through the energy gradient, whose H phi they compute) and the
oracle: f apart from phi, f = phi, in place, off a 16-byte boundary, and captured."""
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


@pytest.mark.parametrize("M", [16, 32, 64, 128, 256])
@pytest.mark.parametrize("off", [0, 1])
def test_one_small_field(G, M, off):
    n, L = (M, M), (7.0, 6.0)
    V = I.harmonic(n, L) + 0.2 * I.smooth_bumps(n, L, 2)
    po = O.Problem(n, L, 31.0, 0.7, V)
    h = L[0] * L[1] * 4.0 / (M * M)

    def put(a):
        t = torch.empty(M * M + off, dtype=torch.complex64, device="cuda")[off:].view(M, M)
        t.copy_(torch.from_numpy(a.astype(np.complex64)))
        return t

    phi, f = put(I.random_field(1, n, L)), put(I.random_field(2, n, L))
    ph, fh = phi.cpu().numpy().astype(complex), f.cpu().numpy().astype(complex)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s), G.Context(n, L, 31.0, 0.7, V, prec=G.GPE_MIXED) as ctx:
        out, grad = torch.empty_like(f), torch.empty_like(f)
        want = O.apply_H(po, ph, fh)
        ctx.apply_H(phi, f, out)
        assert np.max(np.abs(out.cpu().numpy() - want)) <= 2e-5 * np.max(np.abs(want))
        g = f.clone()
        ctx.apply_H(phi, g, g)
        assert torch.equal(g, out)
        ctx.apply_H(phi, phi, out)
        ctx.energy_grad(phi, grad)  # 2 h^d H_phi phi by the passes
        assert float((grad / (2 * h) - out).abs().max()) <= 2e-5 * float(out.abs().max())
        graph = torch.cuda.CUDAGraph()
        got = torch.zeros_like(f)
        with torch.cuda.graph(graph, stream=s):
            ctx.apply_H(phi, phi, got)
        graph.replay()
        s.synchronize()
        assert torch.equal(got, out)
        del graph
