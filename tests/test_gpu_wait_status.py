"""A bounded wait of the dataflow that gives up is an error the host sees: with the
waits set to give up at once (gpe_set_wait_polls(-1)), H phi on a large complex64 field
or batch ends by itself, the next call that returns scalars reports GPE_ERR_TIMEOUT
once, a tangent solve on the broken operator does not return GPE_OK, and with the
default limit the context gives the results it gave before."""
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


def status_of(G, call):
    with pytest.raises(G.GpeError) as e:
        call()
    return e.value.status


def test_field_in_three_dimensions(G):
    n, L = (256, 256, 64), (6.0, 6.0, 6.0)
    phi = I.anisotropic_gaussian(n, L, [1.0, 1.0, 2.0])
    phi = torch.from_numpy(phi).cuda().to(torch.complex64)
    out, ref, z = torch.empty_like(phi), torch.empty_like(phi), torch.empty_like(phi)
    g_rho = torch.ones(phi.shape, dtype=torch.float64, device="cuda")
    g_rho[: 32] = 0.0
    with G.Context(n, L, 10.0, 0.1, I.harmonic(n, L, [1.0, 1.0, 2.0]), prec=G.GPE_MIXED) as ctx:
        ctx.apply_H(phi, phi, ref)
        before = ctx.energy(phi)
        rhs = ref * 1.0j + phi.roll(3, 0)
        ctx.set_wait_polls(-1)
        ctx.apply_H(phi, phi, out)
        assert status_of(G, lambda: ctx.energy(phi)) == G.GPE_ERR_TIMEOUT
        assert ctx.energy(phi) == before  # reported once; energies take no such wait
        ctx.apply_H(phi, phi, out)
        assert status_of(G, lambda: ctx.energy_grad(phi)) == G.GPE_ERR_TIMEOUT
        assert status_of(G, lambda: ctx.tangent_solve(phi, rhs, z, tol=1e-3, max_iter=8)) == G.GPE_ERR_TIMEOUT
        assert status_of(G, lambda: ctx.density_adjoint(phi, g_rho, torch.empty_like(g_rho), tol=1e-3,
                                                        max_iter=8)) == G.GPE_ERR_TIMEOUT
        ctx.set_wait_polls(0)
        ctx.apply_H(phi, phi, out)
        assert ctx.energy(phi) == before and torch.equal(out, ref)


def test_batch(G):
    M, nb = 128, 200
    n, L = (M, M), (8.0, 8.0)
    g = torch.Generator(device="cuda").manual_seed(3)
    f = torch.randn((nb, M, M), dtype=torch.complex64, device="cuda", generator=g)
    out, ref = torch.empty_like(f), torch.empty_like(f)
    with G.Context(n, L, 20.0, 0.4, I.harmonic(n, L), prec=G.GPE_MIXED) as ctx:
        ctx.apply_H_batch(nb, f, f, ref)
        ctx.set_wait_polls(-1)
        ctx.apply_H_batch(nb, f, f, out)
        assert status_of(G, lambda: ctx.energy(f)) == G.GPE_ERR_TIMEOUT
        ctx.set_wait_polls(0)
        ctx.apply_H_batch(nb, f, f, out)
        assert np.isfinite(ctx.energy(f)["total"]) and torch.equal(out, ref)
