"""The scalar steps of a solve on the smallest blocks: grids whose passes run
with fewer than 32 threads per block (one thread sums and steps alone), with
one warp, and with several warps, in 2D and 3D, in the graph and host loops,
each iterate against the FP64 oracle (E_n rel 1e-12, phi_n phase-aligned L2
1e-9 over 6 iterations, the tolerances of the larger grids)."""
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


def _problem(n):
    L = tuple(4.0 + 0.5 * i for i in range(len(n)))
    V = I.harmonic(n, L, [1.0, 1.0, 2.0][:len(n)])
    phi0 = I.perturbed(I.anisotropic_gaussian(n, L, [1.0, 1.0, 2.0][:len(n)]), 3, n, L, 0.05)
    return n, L, 20.0, 0.3, V, phi0


@pytest.mark.parametrize("use_graph", [1, 0])
@pytest.mark.parametrize("n", [(8, 8), (8, 32), (64, 16), (8, 8, 8), (16, 8, 32)])
def test_iterates_on_small_blocks(G, n, use_graph):
    n, L, eta, om, V, phi0 = _problem(n)
    K = 6
    _, orep = O.pcg_solve(O.Problem(n, L, eta, om, V), phi0, O.SolveOptions(max_iter=K), keep_iterates=(K,))
    with G.Context(n, L, eta, om, V, prec=G.GPE_FP64) as ctx:
        phi = torch.from_numpy(phi0.copy()).cuda()
        o = G.solve_opts_default()
        o.max_iter, o.use_graph = K, use_graph
        rep = ctx.pcg_solve(phi, o, log_cap=16)
    assert rep["iters"] == K and rep["log"].shape[0] == K + 1
    for k in range(K + 1):
        e = orep["log"][k]
        assert abs(rep["log"][k, 2] - e["E"]) <= 1e-12 * abs(e["E"]), k
        assert abs(rep["log"][k, 4] - e["res_inf"]) <= 1e-9 * e["res_inf"], k
    a, b = phi.cpu().numpy(), orep["iterates"][K]
    z = np.vdot(a, b)
    assert np.linalg.norm(a * (z / abs(z)) - b) <= 1e-9 * np.linalg.norm(b)


@pytest.mark.parametrize("n", [(8, 8), (16, 32), (8, 16, 8)])
def test_mixed_solve_on_small_blocks(G, n):
    n, L, eta, om, V, phi0 = _problem(n)
    _, orep = O.pcg_solve(O.Problem(n, L, eta, om, V), phi0, O.SolveOptions())
    with G.Context(n, L, eta, om, V, prec=G.GPE_MIXED) as ctx:
        phi = torch.from_numpy(phi0.copy()).cuda()
        rep = ctx.pcg_solve(phi, check=True)
    assert rep["res_inf"] < 1e-8 and abs(rep["E"] - orep["E"]) <= 1e-10 * abs(orep["E"])
