"""Kernels that may start while the one before them in the stream still ends (the
preconditioner's passes, the Thomas-Fermi steps): each call gives the same bits when its
inputs are written by the kernel directly in front of it, when calls follow each other
without a pause on one set of buffers, and when they are captured, as it does on an idle
device."""
import numpy as np
import pytest

from paper_1611_02045_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G(built_lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_02045_gb300 import gpe
    return gpe


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n", [(16, 16), (64, 32), (512, 512), (32, 64, 16), (128, 128, 128)])
def test_chain_gives_the_bits_of_single_calls(G, n, prec):
    L = (7.0, 6.0, 5.0)[:len(n)]
    V = I.harmonic(n, L) + 0.2 * I.smooth_bumps(n, L, 2)
    dt = torch.complex64 if prec == "mixed" else torch.complex128
    g = torch.Generator(device="cuda").manual_seed(3)
    shape = tuple(reversed(n))
    src = [torch.randn(shape, dtype=dt, device="cuda", generator=g) for _ in range(6)]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s), G.Context(n, L, 31.0, 0.3, V,
                                         prec=G.GPE_MIXED if prec == "mixed" else G.GPE_FP64) as ctx:
        phi, r = torch.empty_like(src[0]), torch.empty_like(src[0])
        single = []
        for i in range(6):
            phi.copy_(src[i])
            r.copy_(src[(i + 1) % 6])
            out = torch.empty_like(phi)
            s.synchronize()
            ctx.precond(phi, r, 0.0 if i % 2 else 1.5, out)
            s.synchronize()
            single.append(out)
        tf = torch.empty(shape, dtype=torch.complex128, device="cuda")
        ctx.thomas_fermi(tf)
        s.synchronize()

        def chain(outs, start):
            for i in range(6):  # the copies write the inputs while the call before still ends
                phi.copy_(src[i])
                r.copy_(src[(i + 1) % 6])
                ctx.precond(phi, r, 0.0 if i % 2 else 1.5, outs[i])
                if start is not None:
                    ctx.thomas_fermi(start)

        for _ in range(3):
            outs, start = [torch.zeros_like(phi) for _ in range(6)], torch.zeros_like(tf)
            chain(outs, start)
            s.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(outs, single)) and torch.equal(start, tf)
        outs = [torch.zeros_like(phi) for _ in range(6)]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            chain(outs, None)
        for _ in range(2):
            for o in outs:
                o.zero_()
            graph.replay()
            s.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(outs, single))
        del graph
