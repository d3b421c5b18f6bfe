"""RMS rounding error of the FP64 line transforms: H f of a free particle, one axis
with frequencies that matter (the other axis spans 1e12, where the symbol is nothing
next to a rounding), against the same transforms in extended precision.

The bounds are in units of 2^-53 of the RMS result.  They come from an emulation of
the transforms stage by stage one precision down (binary32 values, fused operations
exact): with twiddles to the nearest number and one multiplication per value and
stage the errors are 1.52 to 2.66, with twiddles from rounded angles and cascaded
butterflies 1.87 to 3.33; each bound is the geometric mean of its two."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOUND = {(16, 8): 1.685, (32, 8): 2.112, (64, 8): 2.264, (128, 8): 2.568, (256, 8): 2.731, (512, 8): 2.866,
         (32, 4): 2.189, (64, 4): 2.332, (128, 4): 2.605, (256, 4): 2.731, (512, 4): 2.974}


@pytest.mark.parametrize("M,E", sorted(BOUND))
@pytest.mark.parametrize("axis", [0, 1])
def test_fp64_transform_pair_rounding(built_lib, M, E, axis):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_02045_gb300 import gpe
    other = 512 if M < 64 else 64
    n, L = ((M, other), (1.0, 1e12)) if axis == 0 else ((other, M), (1e12, 1.0))
    f = np.random.default_rng(M + axis).standard_normal((n[1], n[0], 2)) @ np.array([1.0, 1.0j])
    fd = torch.from_numpy(f).cuda()
    out = torch.empty_like(fd)
    with gpe.Context(n, L, 0.0, 0.0, np.zeros((n[1], n[0])), prec=gpe.GPE_FP64) as ctx:
        ctx.set_plan(1, axis, E, 2)
        ctx.apply_H(fd, fd, out)
        got = out.cpu().numpy().astype(np.clongdouble)
    p = np.where(np.arange(M) < M // 2, np.arange(M), np.arange(M) - M)
    k = (p * np.pi).astype(np.longdouble)
    assert np.finfo(np.longdouble).eps < 1e-18
    dim = 1 - axis  # arrays are [y][x]
    k2 = (k * k / 2)[None, :] if axis == 0 else (k * k / 2)[:, None]
    want = np.fft.ifft(np.fft.fft(f.astype(np.clongdouble), axis=dim) * k2, axis=dim)
    assert want.dtype == np.clongdouble
    err = float(np.sqrt(np.mean(np.abs(got - want) ** 2) / np.mean(np.abs(want) ** 2))) * 2.0**53
    assert err <= BOUND[M, E], err
