"""Thomas-Fermi initial data and spectral interpolation at the edges of what
they accept: potentials on which the root search cannot rely on a smooth mass
(one value everywhere, one deep point, two far levels, random values), the
smallest and flattest grids, and interpolation along each axis alone and all
together, against the oracle's bisection and numpy's FFT."""
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


def _potential(kind, n, L):
    V = I.harmonic(n, L)
    if kind == "flat":
        return np.full(V.shape, 3.25)
    if kind == "deep":
        V.flat[V.size // 3] = -1e6
        return V
    if kind == "levels":
        return np.where(V > np.median(V), 1e4, -2.0)
    if kind == "random":
        return 50.0 * I.uniform_pm1(11, V.size).reshape(V.shape)
    return V


@pytest.mark.parametrize("n", [(8, 8), (512, 8), (128, 64), (8, 16, 32)])
@pytest.mark.parametrize("kind", ["harmonic", "flat", "deep", "levels", "random"])
@pytest.mark.parametrize("eta", [1e-3, 700.0])
def test_thomas_fermi_root(G, n, kind, eta):
    L = tuple(6.0 + i for i in range(len(n)))
    V = _potential(kind, n, L)
    want, mu_o = O.thomas_fermi_state(O.Problem(n, L, eta, 0.0, V))
    out = torch.empty(I.shape_of(n), dtype=torch.complex128, device="cuda")
    with G.Context(n, L, eta, 0.0, V) as ctx:
        mu = ctx.thomas_fermi(out)
        mu2 = ctx.thomas_fermi(out)
    # both roots carry the rounding of a sum of N terms (eps log2 N) relative to mu and V's scale
    scale = abs(mu_o) + np.abs(V).max()
    assert abs(mu - mu_o) <= 1e-13 * scale and mu2 == mu
    phi = out.cpu().numpy()
    assert np.all(phi.imag == 0)
    # |phi|^2 = (mu - V) / eta inherits that error of mu, pointwise
    assert np.max(np.abs(phi.real ** 2 - np.maximum(mu_o - V, 0) / eta)) <= 3e-13 * scale / eta
    assert want.shape == phi.shape


@pytest.mark.parametrize("n,fine", [((8, 8), (16, 8)), ((8, 8), (8, 16)), ((16, 128), (32, 256)), ((256, 8), (512, 16)),
                                    ((8, 16, 8), (8, 16, 16)), ((16, 8, 32), (32, 16, 64))])
def test_interpolation_axes(G, n, fine):
    L = tuple(5.0 for _ in n)
    f = I.random_field(3, n, L)
    want = f
    for ax in range(len(n)):
        if fine[ax] == n[ax]:
            continue
        M, a = n[ax], len(n) - 1 - ax
        F = np.moveaxis(np.fft.fft(want, axis=a), a, -1)
        P = np.zeros(F.shape[:-1] + (2 * M,), dtype=complex)
        P[..., :M // 2] = F[..., :M // 2]
        P[..., -M // 2 + 1:] = F[..., -M // 2 + 1:]
        P[..., M // 2] = P[..., -M // 2] = 0.5 * F[..., M // 2]
        want = np.moveaxis(2.0 * np.fft.ifft(P), -1, a)
    V = I.harmonic
    with G.Context(n, L, 1.0, 0.0, V(n, L)) as c, G.Context(fine, L, 1.0, 0.0, V(fine, L)) as d:
        src = torch.from_numpy(f).cuda()
        dst = torch.full(I.shape_of(fine), float("nan"), dtype=torch.complex128, device="cuda")
        c.interpolate_to(d, src, dst)
    # FP64 transforms: eps times the stages of up to three axes and both directions
    assert np.max(np.abs(dst.cpu().numpy() - want)) <= 2e-14 * np.max(np.abs(want))
