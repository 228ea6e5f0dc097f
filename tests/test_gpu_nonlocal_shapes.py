"""The non-local term at the shapes whose complex64 columns take the warp pass (64 to
512 points, propagation and convolution, 2D and 3D): complex64 against complex128
of the same problem, with samples at the end of the run and without.

complex64 runs are held to 1e-4 at 100 steps; these take 6, where a tenth of that
is ample."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 1e-5


def _run(dtype, shape, npaths, every, noise, steps=6):
    import torch
    from paper_1204_4255_gb300 import xsde
    rng = np.random.default_rng(7)
    ax = [np.linspace(-6.0, 6.0, n, endpoint=False) for n in shape]
    r2 = sum(np.meshgrid(*[x ** 2 for x in ax], indexing="ij"))
    psi0 = np.exp(-0.5 * r2) * np.exp(0.1j * rng.standard_normal((npaths,) + shape))
    off = sum(np.meshgrid(*[(np.fft.fftfreq(n, 1.0 / n) * 12.0 / n) ** 2 for n in shape], indexing="ij"))
    # not even along dimension 0: a transposed or mirrored kernel would show
    skew = np.meshgrid(*[np.fft.fftfreq(n, 1.0 / n) for n in shape], indexing="ij")[0] > 0
    P = xsde.Problem(shape, (-6.0,) * len(shape), (6.0,) * len(shape), dtype)
    P.set_operators(g=2.0, pot_kind=xsde.XSDE_POT_HARMONIC, omega=(1.0,) * len(shape), noise_kind=noise, seed=5,
                    amplitude=0.05 if noise else 0.0)
    P.set_nonlocal(np.fft.fftn((1.0 + 0.5 * skew) / np.sqrt(off + 0.25) * np.prod([12.0 / n for n in shape])))
    pp = torch.zeros((steps // every + 1, npaths, 2), dtype=torch.float64, device="cuda")
    P.moments(every, xsde.XSDE_MOM_NORM | xsde.XSDE_MOM_ENERGY, pp)
    t = torch.from_numpy(psi0.astype(np.complex64)).to(torch.complex64 if dtype == "c64" else torch.complex128).cuda()
    P.integrate(t, 5e-4, steps)
    P.synchronize()
    P.close()
    return t.cpu().numpy(), pp.cpu().numpy()


@pytest.mark.parametrize("shape,npaths", [((256, 64), 3), ((512, 64), 5), ((64, 512), 1), ((512, 16), 1), ((256, 256), 3),
                                          ((64, 16, 16), 3), ((16, 64, 16), 1), ((64, 64, 64), 1), ((16, 128, 64), 1),
                                          ((256, 16, 16), 1), ((16, 16, 64), 3)])
@pytest.mark.parametrize("every", [3, 4])
@pytest.mark.parametrize("noise", [0, 2])
def test_warp_columns_with_the_pair_potential(shape, npaths, every, noise):
    a, pa = _run("c64", shape, npaths, every, noise)
    b, pb = _run("c128", shape, npaths, every, noise)
    assert np.linalg.norm(a - b) / np.linalg.norm(b) < TOL
    assert np.max(np.abs(pa - pb) / np.abs(pb)) < TOL
