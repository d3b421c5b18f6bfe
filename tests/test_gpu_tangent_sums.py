"""The tangent-space solve's grid sums (several inner products per kernel, the
last block's total and scalar step) from fewer points than one block has threads
up to several points per thread: the returned z solves P K z = P rhs, checked
with the oracle's operators, in complex128 and complex64."""
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


@pytest.mark.parametrize("n", [(8, 8), (16, 8), (64, 16), (16, 8, 16), (256, 128)])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_tangent_solve_residual(G, n, prec):
    L = tuple(4.0 for _ in n)
    V = I.harmonic(n, L, [1.0, 1.3, 2.0][:len(n)])
    eta, om = 15.0, 0.2
    po = O.Problem(n, L, eta, om, V)
    phi0 = I.perturbed(I.anisotropic_gaussian(n, L, [1.0, 1.3, 2.0][:len(n)]), 3, n, L)
    phi, rep = O.pcg_solve(po, phi0, O.SolveOptions(tol_res_inf=1e-10))
    assert rep["status"] == "converged"
    dt, tol, bound = (torch.complex128, 1e-11, 1e-9) if prec == 0 else (torch.complex64, 1e-4, 1e-3)
    rhs = I.random_field(8, n, L)
    with G.Context(n, L, eta, om, V, prec=prec) as ctx:
        z = torch.empty(I.shape_of(n), dtype=dt, device="cuda")
        r = ctx.tangent_solve(torch.from_numpy(phi).to("cuda", dt), torch.from_numpy(rhs).to("cuda", dt), z, tol=tol)
        again = torch.empty_like(z)
        r2 = ctx.tangent_solve(torch.from_numpy(phi).to("cuda", dt), torch.from_numpy(rhs).to("cuda", dt), again, tol=tol)
    assert r["status"] == G.GPE_OK and r["rel_res"] <= tol and r2["iters"] == r["iters"]
    assert torch.equal(z, again)  # fixed-order sums
    zz = z.cpu().numpy().astype(complex)
    lam = O.chemical_potential(po, phi)
    proj = lambda h: h - O.inner(po, phi, h) * phi
    Kz = O.apply_H(po, phi, zz) + eta * np.abs(phi) ** 2 * zz + eta * phi ** 2 * zz.conj() - lam * zz
    # the solver's own stopping bound, with room for the operators' rounding in its recurrence
    assert O.norm(po, proj(Kz) - proj(rhs)) <= bound * O.norm(po, proj(rhs))
    assert abs(O.inner(po, phi, zz)) <= bound * O.norm(po, zz)
