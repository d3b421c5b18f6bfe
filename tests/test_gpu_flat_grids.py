"""Sums over many blocks of few threads: grids whose last axis is short, where the pass
that ends an operator runs in blocks of a warp or less by default or by the caller's
plan.  Energies against the oracle (rel 1e-12 complex128, 2e-5 complex64), the same
under the narrowest and the widest plans, and the default call of a flat grid within
four times the time of a cube of the same size (a last block that summed its 1024
partials one load at a time took 5 times as long)."""
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


def widths(n, axis, E):
    """The narrowest and the widest width of a plan (thread cap 256, at most 4096 blocks)."""
    per, outer = (1, int(np.prod(n)) // n[0]) if axis == 0 else (n[0], int(np.prod(n)) // n[0] // n[axis])
    ok = [w for w in (1 << k for k in range(10)) if w * n[axis] // E <= 256 and w <= (outer if axis == 0 else per)
          and (outer // w if axis == 0 else per // w * outer) <= 4096]
    return ok[0], ok[-1]


@pytest.mark.parametrize("n", [(16, 8), (8, 8), (512, 8), (128, 128, 8), (8, 64, 8), (16, 8, 64), (256, 64, 16), (64, 8, 16)])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_energy_on_flat_grids(G, n, prec):
    L = (5.0, 6.0, 7.0)[: len(n)]
    V = I.harmonic(n, L)
    dt, tol = (torch.complex128, 1e-12) if prec == 0 else (torch.complex64, 2e-5)
    phi = torch.from_numpy(np.ascontiguousarray(I.random_field(3, n, L))).cuda().to(dt)
    po = O.Problem(n, L, 9.0, 0.5, V)
    ph = phi.cpu().numpy().astype(complex)
    want_E, want_lam = O.energy(po, ph), O.chemical_potential(po, ph)
    with G.Context(n, L, 9.0, 0.5, V, prec=prec) as ctx:
        plans = [None] + [[(8, widths(n, ax, 8)[i]) for ax in range(len(n))] for i in (0, 1)]
        for p in plans:
            for ax in range(len(n) if p else 0):
                ctx.set_plan(1 if prec == 0 else 0, ax, *p[ax])
            e = ctx.energy(phi)
            assert abs(e["total"] - want_E) <= tol * abs(want_E), p
            assert abs(e["lam"] - want_lam) <= tol * abs(want_lam), p


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_flat_grids_sum_as_fast_as_cubes(G, prec):
    def best(n):
        L = (8.0, 8.0, 8.0)
        dt = torch.complex128 if prec == 0 else torch.complex64
        phi = torch.randn(I.shape_of(n), dtype=dt, device="cuda")
        times = []
        with G.Context(n, L, 9.0, 0.5, I.harmonic(n, L), prec=prec) as ctx:
            for _ in range(30):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                ctx.energy(phi)
                b.record()
                b.synchronize()
                times.append(a.elapsed_time(b))
        return min(times)
    flat, cube = best((128, 128, 8)), best((64, 64, 32))
    assert flat <= 4.0 * cube, (flat, cube)
