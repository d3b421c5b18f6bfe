"""The default plans of the pass kernels (E and width per launch mode and axis,
chosen from the grid's size) on square, cubic, flat and tiny grids: every one
is a plan that gpe_set_plan accepts for that grid, and H phi, P_C r and the
energy under the defaults match the oracle (rel 1e-12 in complex128, 2e-5 in
complex64, as everywhere)."""
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


GRIDS = [(8, 8), (8, 512), (512, 8), (16, 32), (64, 512), (512, 256), (512, 512), (8, 8, 512), (512, 8, 8),
         (16, 16, 256), (32, 32, 32), (64, 64, 32), (64, 64, 64)]  # both sides of 2^17 points


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_default_plans(G, n, prec):
    L = tuple(6.0 + i for i in range(len(n)))
    V = I.harmonic(n, L)
    eta, om = 23.0, 0.6
    po = O.Problem(n, L, eta, om, V)
    dt, tol = (torch.complex128, 1e-12) if prec == 0 else (torch.complex64, 2e-5)
    phi = torch.from_numpy(I.random_field(1, n, L)).to("cuda", dt)
    f = torch.from_numpy(I.random_field(2, n, L)).to("cuda", dt)
    out = torch.empty_like(f)
    with G.Context(n, L, eta, om, V, prec=prec) as ctx:
        for mode in ([1] if prec == 0 else [0, 1, 2]):
            for ax in range(len(n)):
                E, w = ctx.get_plan(mode, ax)
                ctx.set_plan(mode, ax, E, w)
                assert ctx.get_plan(mode, ax) == (E, w)
        ph, fh = phi.cpu().numpy().astype(complex), f.cpu().numpy().astype(complex)
        ctx.apply_H(phi, f, out)
        want = O.apply_H(po, ph, fh)
        assert np.max(np.abs(out.cpu().numpy() - want)) <= tol * np.max(np.abs(want))
        ctx.precond(phi, f, 0.0, out)
        want = O.precond_C(po, ph, fh, O.lambda_tilde(po, ph))
        assert np.max(np.abs(out.cpu().numpy() - want)) <= tol * np.max(np.abs(want))
        e = ctx.energy(phi)
        assert abs(e["total"] - O.energy(po, ph)) <= (1e-12 if prec == 0 else 2e-6) * abs(O.energy(po, ph))
