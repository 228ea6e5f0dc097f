"""Norm and energy samples at the ends of the number range, fields that do not depend on
being sampled, and paths in ensembles of different sizes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(shape, dtype, g, basis=(), scheme=0, noise=0, variant=0):
    from paper_1204_4255_gb300 import xsde
    lo = tuple(0.0 if basis and basis[d] else -6.0 for d in range(len(shape)))
    P = xsde.Problem(shape, lo, (6.0,) * len(shape), dtype, basis=basis)
    P.set_operators(g=g, pot_kind=xsde.XSDE_POT_HARMONIC if shape else xsde.XSDE_POT_NONE, omega=(1.0,) * len(shape),
                    noise_kind=noise, seed=9, amplitude=0.02 if noise else 0.0)
    if scheme:
        xsde.xsde_set_scheme(P.prob, scheme)
    if variant:
        xsde.xsde_set_kernel_variant(P.prob, variant)
    return P


def _field(shape, npaths, seed=1):
    rng = np.random.default_rng(seed)
    ax = [np.linspace(-6.0, 6.0, n, endpoint=False) for n in shape]
    r2 = sum(np.meshgrid(*[x ** 2 for x in ax], indexing="ij"))
    return np.exp(-0.3 * r2) * np.exp(0.2j * rng.standard_normal((npaths,) + shape))


def _samples(shape, dtype, g, psi, steps=2, every=1, **more):
    import torch
    from paper_1204_4255_gb300 import xsde
    P = _problem(shape, dtype, g, **more)
    pp = torch.zeros((steps // every + 1, len(psi), 2), dtype=torch.float64, device="cuda") if every else None
    if every:
        P.moments(every, xsde.XSDE_MOM_NORM | xsde.XSDE_MOM_ENERGY, pp)
    t = torch.from_numpy(np.ascontiguousarray(psi)).to(torch.complex64 if dtype == "c64" else torch.complex128).cuda()
    P.integrate(t, 1e-4, steps)
    P.synchronize()
    P.close()
    return t.cpu().numpy(), pp.cpu().numpy() if every else None


@pytest.mark.parametrize("shape", [(64,), (512,), (32, 64), (16, 16, 32)])
def test_energy_of_large_linear_fields(shape):
    """without a nonlinearity the energy is quadratic in the field: 1e100 times the
    field has 1e200 times the energy (|psi|^4 leaves FP64's range there)"""
    psi = _field(shape, 2)
    _, one = _samples(shape, "c128", 0.0, psi)
    _, big = _samples(shape, "c128", 0.0, psi * 2.0 ** 332)
    assert np.isfinite(big).all()
    assert np.allclose(big * 2.0 ** -664, one, rtol=1e-12, atol=0)


@pytest.mark.parametrize("shape", [(64,), (1024,), (16, 16), (64, 128), (64, 512), (16, 32, 64)])
def test_norm_of_small_complex64_fields(shape):
    """|psi|^2 near 1e-40 is a whole number of 2^-149; each point's is off by at most
    two halves (its squares' and their sum's rounding) and then counts in full"""
    amp = 2.0 ** -66
    psi = (_field(shape, 2) * amp).astype(np.complex64).astype(np.complex128)
    _, pp = _samples(shape, "c64", 0.0, psi)
    want = (np.abs(psi) ** 2).reshape(2, -1).sum(1) * np.prod([12.0 / n for n in shape])
    # and the steps leave the norm within 1e-5
    tol = np.prod(shape) * 1.5 * 2.0 ** -149 * np.prod([12.0 / n for n in shape]) / want + 1e-5
    assert (np.abs(pp[:, :, 0] / want - 1.0) < tol).all(), (pp[:, :, 0], want)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("shape", [(64,), (512,), (16, 64), (64, 256), (128, 128), (16, 32, 64)])
def test_sampling_leaves_the_field_alone(shape, dtype):
    psi = _field(shape, 3)
    seen, _ = _samples(shape, dtype, 2.0, psi, steps=4, every=2)
    unseen, _ = _samples(shape, dtype, 2.0, psi, steps=4, every=0)
    assert np.array_equal(seen, unseen)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("shape", [(64, 64), (64, 256), (32, 1024), (16, 32, 128)])
def test_first_sample_leaves_a_semi_implicit_field_alone(shape, dtype):
    psi = _field(shape, 2)
    seen, _ = _samples(shape, dtype, 2.0, psi, steps=3, every=5, scheme=1)
    unseen, _ = _samples(shape, dtype, 2.0, psi, steps=3, every=0, scheme=1)
    assert np.array_equal(seen, unseen)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("shape,npaths,basis,variant", [((32,), 3000, (), 4), ((64,), 12000, (), 4), ((256,), 3000, (), 1),
                                                        ((512,), 320, (), 5), ((1024,), 310, (), 4), ((128, 64), 40, (1, 0), 3),
                                                        ((256, 128), 20, (2, 0), 3), ((64, 64), 32, (), 0)])
def test_a_path_and_the_ensemble_it_runs_in(shape, npaths, basis, variant, dtype):
    """Variant 0 takes its launch shape by the number of paths too, so a path alone and
    in a large ensemble agree to rounding (two steps, each within 1e-6 or 1e-14); with a
    variant set, and on Fourier lattices of 2D, bit for bit."""
    psi = _field(shape, 4)
    many = np.tile(psi, (npaths // 4,) + (1,) * len(shape))
    for v in {0, variant}:
        whole, _ = _samples(shape, dtype, 2.0, many, every=0, basis=basis, variant=v)
        part, _ = _samples(shape, dtype, 2.0, psi, every=0, basis=basis, variant=v)
        for got in (whole[:4], whole[-4:]):
            assert np.linalg.norm(got - part) <= (1e-6 if dtype == "c64" else 1e-14) * np.linalg.norm(part)
            if v or (len(shape) > 1 and not basis):
                assert np.array_equal(got, part)
