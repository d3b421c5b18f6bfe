"""Plans set by the caller are the ones gpe_apply_H runs: on complex64 fields whose
default form is not the passes (small squares, large 3D fields), E = 8 and E = 4 sum
in different orders and so give different bits, both within the complex64 tolerance
(rel 2e-5) of the default form's result; a z plan alone leaves the dataflow in place,
and after gpe_autotune the default form runs again."""
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


def close(a, b):
    return float((a - b).abs().max()) <= 2e-5 * float(b.abs().max())


@pytest.mark.parametrize("n,widths", [((32, 32), (8, 8)), ((64, 64), (4, 4)), ((128, 128), (2, 4)),
                                      ((128, 64, 512), (16, 16)), ((256, 128, 128), (8, 8))])
def test_caller_plans_reach_apply_H(G, n, widths):
    L = tuple(6.0 + i for i in range(len(n)))
    V = I.harmonic(n, L)
    g = torch.Generator(device="cuda").manual_seed(5)
    phi, f = (torch.randn(I.shape_of(n), dtype=torch.complex64, device="cuda", generator=g) for _ in range(2))
    out = [torch.full_like(f, float("nan")) for _ in range(5)]
    with G.Context(n, L, 11.0, 0.7, V, prec=G.GPE_MIXED) as ctx:
        ctx.apply_H(phi, f, out[0])
        if len(n) == 3:
            ctx.set_plan(0, 2, *ctx.get_plan(0, 2))
            ctx.apply_H(phi, f, out[4])
            assert torch.equal(out[4], out[0])
        for k, E in ((1, 8), (2, 4)):
            for axis in (0, 1):
                ctx.set_plan(0, axis, E, widths[axis])
            ctx.apply_H(phi, f, out[k])
            assert close(out[k], out[0]), E
        assert not torch.equal(out[1], out[2])
        if len(n) == 2:
            ctx.autotune(iters=2)
            ctx.apply_H(phi, f, out[3])
            assert torch.equal(out[3], out[0])
