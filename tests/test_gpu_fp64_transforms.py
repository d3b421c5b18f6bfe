"""FP64 line transforms of every length and radix split (E = 8 and 4 values per
thread; fused radix-2, -4 and -8 butterflies after the first stage), along x and
along y, against the oracle.  The bound is the transforms' rounding, eps times
the stages of both directions, relative to the largest result; random fields and
smooth ones (small high-frequency parts next to large low-frequency ones)."""
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


@pytest.mark.parametrize("M", [8, 16, 32, 64, 128, 256, 512])
@pytest.mark.parametrize("axis", [0, 1])
def test_fp64_operators_by_length(G, M, axis):
    n = (M, 16) if axis == 0 else (16, M)
    L = (7.0, 6.0)
    V = I.harmonic(n, L)
    eta, om, alpha = 5.0, 0.8, 0.7
    po = O.Problem(n, L, eta, om, V)
    tol = 8 * np.finfo(float).eps * np.log2(M * 16)
    with G.Context(n, L, eta, om, V, prec=G.GPE_FP64) as ctx:
        for E in (8, 4) if M >= 32 else (8,):
            ctx.set_plan(1, axis, E, 2)
            for phi, f in ((I.random_field(1, n, L), I.random_field(2, n, L)), (I.phi_d(n, L, 0.4), I.phi_a(n, L))):
                ph, fd = torch.from_numpy(phi).cuda(), torch.from_numpy(f).cuda()
                out = torch.empty_like(fd)
                ctx.apply_H(ph, fd, out)
                want = O.apply_H(po, phi, f)
                # the symbol multiplies the operand's rounding by up to max |k|^2 / 2 + ...
                k2 = sum((0.5 * m * np.pi / l) ** 2 for m, l in zip(n, L))
                scale = np.max(np.abs(want)) + (0.5 * k2 + om * max(L) * np.sqrt(k2)) * np.max(np.abs(f))
                assert np.max(np.abs(out.cpu().numpy() - want)) <= tol * scale, E
                ctx.precond(ph, fd, alpha, out)
                want = O.precond_C(po, phi, f, alpha)
                assert np.max(np.abs(out.cpu().numpy() - want)) <= tol * np.max(np.abs(f)) / alpha, E
