"""The dataflow form of H phi on complex64 planes (3D fields of at least 2^22
points, large 2D batches) against the general path, over every pair of sides it
takes, with f = phi and f != phi, in place, in ragged batches, and under stream
capture.  The general path is the same call on fields 8 bytes off a 16-byte
boundary, which the dataflow does not take; both must agree to the complex64
tolerance (rel 2e-5), and samples are checked against the oracle."""
import numpy as np
import pytest

from oracle import gpe_oracle as O
from paper_1611_02045_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
C64 = torch.complex64


@pytest.fixture(scope="module")
def G(built_lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_02045_gb300 import gpe
    return gpe


def field(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, dtype=C64, device="cuda", generator=g)


def off_boundary(x):
    y = torch.empty(x.numel() + 1, dtype=x.dtype, device=x.device)[1:].view(x.shape)
    y.copy_(x)
    assert y.data_ptr() % 16 == 8
    return y


def close(a, b):
    return float((a - b).abs().max()) <= 2e-5 * float(b.abs().max())


@pytest.mark.parametrize("n", [(mx, my, max(16, (1 << 22) // (mx * my))) for mx in (64, 128, 256)
                               for my in (64, 128, 256) if (mx, my) != (64, 64)])
def test_3d_planes_match_the_passes(G, n):
    L = (5.0, 6.0, 7.0)
    V = I.harmonic(n, L, [1.0, 1.2, 2.0]) + 0.3 * I.uniform_pm1(3, int(np.prod(n))).reshape(I.shape_of(n))
    phi, f = field(I.shape_of(n), 1), field(I.shape_of(n), 2)
    phi_o, f_o = off_boundary(phi), off_boundary(f)
    with G.Context(n, L, 11.0, 0.7, V, prec=G.GPE_MIXED) as ctx:
        out, want = torch.full_like(f, float("nan")), torch.empty_like(f)
        for a, b, ao, bo in ((phi, f, phi_o, f_o), (phi, phi, phi_o, phi_o)):
            ctx.apply_H(ao, bo, want)
            for _ in range(2):
                out.fill_(float("nan"))
                ctx.apply_H(a, b, out)
                assert close(out, want)
        g = f.clone()
        ctx.apply_H(phi, g, g)  # in place
        ctx.apply_H(phi_o, f_o, want)
        assert close(g, want)


def test_3d_planes_match_the_oracle(G):
    n, L = (256, 64, 256), (5.0, 6.0, 7.0)
    V = I.harmonic(n, L)
    phi, f = field(I.shape_of(n), 4), field(I.shape_of(n), 5)
    out = torch.empty_like(f)
    with G.Context(n, L, 11.0, 0.7, V, prec=G.GPE_MIXED) as ctx:
        ctx.apply_H(phi, f, out)
        want = O.apply_H(O.Problem(n, L, 11.0, 0.7, V), phi.cpu().numpy().astype(complex), f.cpu().numpy().astype(complex))
        assert np.max(np.abs(out.cpu().numpy() - want)) <= 2e-5 * np.max(np.abs(want))
        # captured: no allocation, the same result from a replay
        s = torch.cuda.Stream()
    with torch.cuda.stream(s), G.Context(n, L, 11.0, 0.7, V, prec=G.GPE_MIXED) as ctx:
        got = torch.zeros_like(f)
        ctx.apply_H(phi, f, got)
        s.synchronize()
        ref = got.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            ctx.apply_H(phi, f, got)
        got.zero_()
        graph.replay()
        s.synchronize()
        assert torch.equal(got, ref)
        del graph


@pytest.mark.parametrize("M,nb", [(64, 768), (64, 1531), (128, 192), (128, 333), (256, 32), (256, 77)])
def test_batches_match_the_clusters(G, M, nb):
    n, L = (M, M), (8.0, 8.0)
    V = I.harmonic(n, L) + 0.2 * I.smooth_bumps(n, L, 3)
    po = O.Problem(n, L, 41.0, 0.6, V)
    phi, f = field((nb, M, M), 7), field((nb, M, M), 8)
    phi_o, f_o = off_boundary(phi), off_boundary(f)
    with G.Context(n, L, 41.0, 0.6, V, prec=G.GPE_MIXED) as ctx:
        out, want = torch.empty_like(f), torch.empty_like(f)
        for a, b, ao, bo in ((phi, f, phi_o, f_o), (f, f, f_o, f_o)):
            out.fill_(float("nan"))
            ctx.apply_H_batch(nb, a, b, out)
            ctx.apply_H_batch(nb, ao, bo, want)
            assert close(out, want)
            for k in (0, nb // 2, nb - 1):
                w = O.apply_H(po, a[k].cpu().numpy().astype(complex), b[k].cpu().numpy().astype(complex))
                assert np.max(np.abs(out[k].cpu().numpy() - w)) <= 2e-5 * np.max(np.abs(w))


def test_batch_larger_than_the_counters_under_capture(G):
    """A batch that outgrows the counters is not allocated for inside a capture:
    the clusters run, and the same batch outside the capture takes the dataflow."""
    M, nb = 64, 1100
    n, L = (M, M), (8.0, 8.0)
    s = torch.cuda.Stream()
    f = field((nb, M, M), 9)
    torch.cuda.synchronize()
    with torch.cuda.stream(s), G.Context(n, L, 30.0, 0.4, I.harmonic(n, L), prec=G.GPE_MIXED) as ctx:
        small = torch.empty_like(f[:8])
        ctx.apply_H_batch(8, f, f, small)  # the clusters' attributes are set before the capture
        out = torch.zeros_like(f)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            ctx.apply_H_batch(nb, f, f, out)
        graph.replay()
        s.synchronize()
        ref = torch.empty_like(f)
        ctx.apply_H_batch(nb, f, f, ref)
        s.synchronize()
        assert close(out, ref)
        del graph


def test_captured_batch_outlives_a_growth_of_the_counters(G):
    """A batch captured with the context's first counters, replayed after a larger batch
    has outgrown them: the same bits as before."""
    M, nb, more = 64, 800, 1100
    n, L = (M, M), (8.0, 8.0)
    s = torch.cuda.Stream()
    f = field((more, M, M), 10)
    torch.cuda.synchronize()
    with torch.cuda.stream(s), G.Context(n, L, 30.0, 0.4, I.harmonic(n, L), prec=G.GPE_MIXED) as ctx:
        out, ref, big = torch.zeros_like(f[:nb]), torch.empty_like(f[:nb]), torch.empty_like(f)
        ctx.apply_H_batch(nb, f[:nb], f[:nb], ref)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            ctx.apply_H_batch(nb, f[:nb], f[:nb], out)
        ctx.apply_H_batch(more, f, f, big)
        graph.replay()
        s.synchronize()
        assert torch.equal(out, ref) and torch.equal(big[:nb], ref)
        del graph
