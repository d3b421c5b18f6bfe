"""The dataflow form of gpe_apply_H_batch at the sizes where it runs (from 2^21 points
at 256^2, 3 2^20 at 64^2 and 128^2): an operand or a result 8 bytes off a 16-byte
boundary, each by itself, goes to the clusters, a density field off the boundary does
not, and ragged batches around the lag between a field's row and column units are
right field by field.  The two forms round their multipliers differently, so equal bits
tell that the same form ran and different bits that another one did."""
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


def off(x):
    y = torch.empty(x.numel() + 1, dtype=x.dtype, device=x.device)[1:].view(x.shape)
    y.copy_(x)
    assert y.data_ptr() % 16 == 8
    return y


def check(po, got, phi, f, fields):
    for k in fields:
        want = O.apply_H(po, phi[k].cpu().numpy().astype(complex), f[k].cpu().numpy().astype(complex))
        assert np.max(np.abs(got[k].cpu().numpy() - want)) <= 2e-5 * np.max(np.abs(want)), k


@pytest.mark.parametrize("M,nb", [(64, 768), (128, 192), (256, 32)])
@pytest.mark.parametrize("what", ["f", "out", "phi"])
def test_each_operand_off_the_boundary(G, M, nb, what):
    n, L = (M, M), (8.0, 8.0)
    V = I.harmonic(n, L) + 0.2 * I.smooth_bumps(n, L, 3)
    phi, f = field((nb, M, M), 1), field((nb, M, M), 2)
    args = dict(phi=phi, f=f, out=torch.full_like(f, float("nan")))
    ref = torch.full_like(f, float("nan"))
    with G.Context(n, L, 41.0, 0.6, V, prec=G.GPE_MIXED) as ctx:
        ctx.apply_H_batch(nb, phi, f, ref)
        args[what] = off(args[what])
        ctx.apply_H_batch(nb, args["phi"], args["f"], args["out"])
        assert torch.equal(args["out"], ref) == (what == "phi")
    check(O.Problem(n, L, 41.0, 0.6, V), args["out"], phi, f, (0, nb // 3, nb - 1))


@pytest.mark.parametrize("nb", [32, 33, 70])
def test_ragged_batches_above_the_threshold(G, nb):
    M = 256
    n, L = (M, M), (16.0, 16.0)
    V = I.harmonic(n, L) + 0.3 * I.smooth_bumps(n, L, 4)
    f = field((nb, M, M), 4)
    out, clusters = torch.full_like(f, float("nan")), torch.full_like(f, float("nan"))
    with G.Context(n, L, 900.0, 0.85, V, prec=G.GPE_MIXED) as ctx:
        ctx.apply_H_batch(nb, f, f, out)
        ctx.apply_H_batch(nb, off(f), off(f), clusters)
    assert not torch.equal(out, clusters)  # the dataflow ran
    check(O.Problem(n, L, 900.0, 0.85, V), out, f, f, range(nb))
