"""complex128 transforms in fixed point: free evolution against long-double FFTs.

With g = 0 and no potential a step is D(D(a)), four transforms a dimension.  An
FP64 FFT of n points stays within u log2 n of the exact one (u = 2^-53, relative
2-norm), so four of them, with their two factors, are held to 4 u log2 n, and a 2D
step to the sum over its dimensions.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
LD, CLD = np.longdouble, np.clongdouble


def _field(kind, shape, seed=3):
    rng = np.random.default_rng(seed)
    if kind == "noise":
        return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    j = np.arange(shape[-1])
    line = np.exp(2j * np.pi * 3 * j / shape[-1]) if kind == "mode" else \
        np.exp(-0.5 * ((j - shape[-1] / 2) * 16.0 / shape[-1]) ** 2) + 0j
    return np.broadcast_to(line, shape).copy()


def _free(psi, box, c0, c2, dt):
    """exp(L dt) psi in long double over the trailing dimensions."""
    if np.finfo(LD).eps > 1e-18:
        pytest.skip("no long double wider than FP64")
    a = psi.astype(CLD)
    for d in range(1, psi.ndim):
        n = psi.shape[d]
        j = np.where(np.arange(n) < n // 2, np.arange(n), np.arange(n) - n).astype(LD)
        k = 2 * LD("3.14159265358979323846264338327950288") / (2 * LD(box)) * j
        E = np.exp((CLD(c0) * (d == 1) + CLD(c2) * k * k) * LD(dt))
        E = E.reshape([-1 if q == d else 1 for q in range(psi.ndim)])
        a = np.fft.ifft(np.fft.fft(a, axis=d) * E, axis=d)
    return a


def _run(psi, box, c0, c2, dt, variant=0):
    import torch
    from paper_1204_4255_gb300 import xsde
    shape = psi.shape[1:]
    P = xsde.Problem(shape, (-box,) * len(shape), (box,) * len(shape), "c128")
    P.set_operators(c0=c0, c2=c2)
    xsde.xsde_set_kernel_variant(P.prob, variant)
    t = torch.from_numpy(psi.astype(np.complex128)).cuda()
    P.integrate(t, dt, 1)
    P.synchronize()
    P.close()
    return t.cpu().numpy()


def _rel(got, ref):
    with np.errstate(under="ignore"):
        s = LD(1) / np.abs(ref).max()
        return float(np.sqrt((np.abs(got.astype(CLD) * s - ref * s) ** 2).sum() / (np.abs(ref * s) ** 2).sum()))


@pytest.mark.parametrize("variant", [0, 1, 4, 5, 6])
@pytest.mark.parametrize("n", [16, 128, 256, 512, 2048])
@pytest.mark.parametrize("kind,scale", [("noise", 1.0), ("mode", 1e150), ("gauss", 1e-290)])
def test_free_lines_are_as_exact_as_fp64(n, variant, kind, scale):
    psi = _field(kind, (3, n)) * scale
    assert _rel(_run(psi, 10.0, 0j, -0.5j, 1e-4, variant), _free(psi, 10.0, 0j, -0.5j, 1e-4)) < 4 * U * np.log2(n)


@pytest.mark.parametrize("shape", [(16, 2048), (512, 32), (64, 256), (1024, 16)])
@pytest.mark.parametrize("kind", ["noise", "gauss"])
def test_free_planes_are_as_exact_as_fp64(shape, kind):
    psi = _field(kind, (2,) + shape)
    assert _rel(_run(psi, 10.0, 0j, -0.5j, 1e-4), _free(psi, 10.0, 0j, -0.5j, 1e-4)) < 4 * U * np.log2(np.prod(shape))


@pytest.mark.parametrize("c0,c2", [(-700.0 + 0j, -0.5j), (0j, -0.5 + 0j), (20.0 + 3j, -0.5j)])
@pytest.mark.parametrize("shape", [(256,), (64, 128)])
def test_damped_and_growing_factors(shape, c0, c2):
    """uniform damping and growth ride on the limbs' exponent; factors spread over
    the spectrum keep FP64 products.  exp(c dt) itself is rounded: its argument,
    up to |c| dt, adds |c dt| u."""
    psi = _field("noise", (2,) + shape)
    dt = 0.05
    k2 = len(shape) * (np.pi / 20.0 * max(shape)) ** 2
    tol = (4 * np.log2(np.prod(shape)) + 4 * dt * (abs(c0) + abs(c2) * k2)) * U
    assert _rel(_run(psi, 20.0, c0, c2, dt), _free(psi, 20.0, c0, c2, dt)) < tol


@pytest.mark.parametrize("shape", [(256,), (32, 64)])
def test_zero_lines_stay_zero_and_nan_lines_spread(shape):
    psi = _field("noise", (3,) + shape)
    psi[1] = 0.0
    psi[(2,) + (5,) * len(shape)] = np.nan
    got = _run(psi, 10.0, 0j, -0.5j, 1e-3)
    assert np.isfinite(got[0]).all() and not got[1].any() and np.isnan(got[2]).all()
