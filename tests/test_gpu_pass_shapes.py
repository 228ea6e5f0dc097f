"""The complex64 passes at the edges of their shapes against the generic passes
(kernel variant 1): 64-point lines and columns, path counts that leave a group of
column warps or a row item without work, cosine / sine columns on the warp pass.

Both run the same scheme in FP32; after `steps` steps each is within the
framework's 1e-5 per 10 steps of the exact field (relative 2-norm, 1e-4 at 100
steps being the acceptance bar of whole runs), so they differ by at most twice that.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 2e-5


def _run(shape, npaths, variant, basis=(), noise=0, scheme=0, nonlocal_=False, every=0, steps=6):
    import torch
    from paper_1204_4255_gb300 import xsde
    rng = np.random.default_rng(7)
    lo = tuple(0.0 if basis and basis[d] else -6.0 for d in range(len(shape)))
    axes = [lo[d] + (np.arange(n) + (0.5 if lo[d] == 0.0 else 0.0)) * (6.0 - lo[d]) / n for d, n in enumerate(shape)]
    r2 = sum(np.meshgrid(*[x ** 2 for x in axes], indexing="ij"))
    psi0 = np.exp(-0.5 * r2) * np.exp(0.1j * rng.standard_normal((npaths,) + shape))
    P = xsde.Problem(shape, lo, (6.0,) * len(shape), "c64", basis=basis)
    P.set_operators(g=2.0, pot_kind=xsde.XSDE_POT_HARMONIC, omega=(1.0,) * len(shape), noise_kind=noise, seed=5,
                    amplitude=0.05 if noise else 0.0)
    if scheme:
        xsde.xsde_set_scheme(P.prob, scheme)
    if nonlocal_:
        P.set_nonlocal(np.fft.fftn(0.01 / (1.0 + np.fft.ifftshift(r2))))
    if xsde.xsde_kernel_variants(P.prob) > 1:
        xsde.xsde_set_kernel_variant(P.prob, variant)
    pp = torch.zeros((steps // every + 1, npaths, 2), dtype=torch.float64, device="cuda") if every else None
    if every:
        P.moments(every, xsde.XSDE_MOM_NORM | xsde.XSDE_MOM_ENERGY, pp)
    t = torch.from_numpy(psi0.astype(np.complex64)).cuda()
    P.integrate(t, 5e-4, steps)
    P.synchronize()
    P.close()
    return t.cpu().numpy(), pp.cpu().numpy() if every else None


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("shape,npaths", [((64, 64), 1), ((16, 64), 3), ((64, 1024), 1), ((512, 64), 7), ((128, 128), 5),
                                          ((256, 512), 3), ((512, 256), 1), ((64, 64, 64), 1), ((16, 128, 64), 3)])
@pytest.mark.parametrize("noise", [0, 1, 2])
def test_fast_passes_match_generic(shape, npaths, noise):
    a, pa = _run(shape, npaths, 0, noise=noise, every=3)
    b, pb = _run(shape, npaths, 1, noise=noise, every=3)
    assert _rel(a, b) < TOL and np.max(np.abs(pa - pb) / np.abs(pb)) < TOL


@pytest.mark.parametrize("shape,npaths,basis", [((128, 64), 25, (1, 0)), ((256, 128), 13, (2, 0)), ((256, 16), 90, (1, 0)),
                                                ((16, 128, 32), 2, (0, 1, 0)), ((128, 16, 64), 1, (2, 0, 0))])
def test_cosine_sine_columns_match_generic(shape, npaths, basis):
    a, pa = _run(shape, npaths, 0, basis=basis, every=3)
    b, pb = _run(shape, npaths, 1, basis=basis, every=3)
    assert _rel(a, b) < TOL and np.max(np.abs(pa - pb) / np.abs(pb)) < TOL


@pytest.mark.parametrize("shape,npaths", [((64, 64), 3), ((16, 128), 1), ((512, 64), 1), ((128, 1024), 2), ((64, 64, 64), 1),
                                          ((16, 32, 128), 3)])
@pytest.mark.parametrize("every", [0, 2, 3])
def test_semi_implicit_rows_match_complex128(shape, npaths, every):
    """one shape of the scheme: against complex128 of the same problem"""
    import torch
    from paper_1204_4255_gb300 import xsde
    rng = np.random.default_rng(3)
    x = [np.linspace(-6, 6, n, endpoint=False) for n in shape]
    psi0 = np.exp(-0.5 * sum(np.meshgrid(*[v ** 2 for v in x], indexing="ij"))) * \
        np.exp(0.1j * rng.standard_normal((npaths,) + shape))
    out = []
    for name, cd in (("c64", torch.complex64), ("c128", torch.complex128)):
        P = xsde.Problem(shape, (-6.0,) * len(shape), (6.0,) * len(shape), name)
        P.set_operators(g=2.0, pot_kind=xsde.XSDE_POT_HARMONIC, omega=(1.0,) * len(shape),
                        noise_kind=xsde.XSDE_NOISE_WIENER_COMPLEX, seed=5, amplitude=0.05)
        xsde.xsde_set_scheme(P.prob, xsde.XSDE_SCHEME_SEMI_IMPLICIT)
        pp = torch.zeros((6 // max(every, 1) + 1, npaths, 2), dtype=torch.float64, device="cuda")
        if every:
            P.moments(every, xsde.XSDE_MOM_NORM | xsde.XSDE_MOM_ENERGY, pp)
        t = torch.from_numpy(psi0).to(cd).cuda()
        P.integrate(t, 5e-4, 6)
        P.synchronize()
        P.close()
        out.append((t.cpu().numpy(), pp.cpu().numpy()))
    assert _rel(out[0][0], out[1][0]) < TOL
    if every:
        assert np.max(np.abs(out[0][1] - out[1][1]) / np.abs(out[1][1])) < TOL
