"""The scale of complex128 lines in fixed point (csrc/fx.cuh) where it is tightest:
components just above the bottom of a binade, -(1 - d) 2^k, on whole lines.

Tolerances as in test_gpu_fixed_point.py: a free step is four transforms a
dimension, each within u log2 n of the exact one.
"""
import numpy as np
import pytest

from test_gpu_fixed_point import _field, _free, _rel, _run, CLD, U

pytestmark = pytest.mark.gpu

OFFSETS = [0.0, 2.0 ** -53, 1e-10, 2.0 ** -28]


def _check(psi, variant=0):
    got = _run(psi, 10.0, 0j, -0.5j, 1e-4, variant)
    ref = _free(psi[:1], 10.0, 0j, -0.5j, 1e-4)   # every path holds the same field
    for p in {0, len(psi) // 2, len(psi) - 1}:
        assert _rel(got[p:p + 1], ref) < 4 * U * np.log2(np.prod(psi.shape[1:]))


@pytest.mark.parametrize("re,im", [(-1.0, -1.0), (-1.0, 1.0), (1.0, -1.0)])
@pytest.mark.parametrize("d", OFFSETS)
@pytest.mark.parametrize("npaths,shape,variant", [(3, (512,), 1), (400, (512,), 0), (2, (2048,), 6), (2, (16,), 1), (2, (64,), 1),
                                                  (3, (256,), 0), (2, (16, 16), 0), (2, (64, 512), 0), (1, (256, 32), 0),
                                                  (1, (16, 32, 64), 0)])
def test_lines_at_the_bottom_of_a_binade(npaths, shape, variant, d, re, im):
    for k in (0, -3, 40):
        _check(np.full((npaths,) + shape, (1.0 - d) * complex(re, im) * 2.0 ** k), variant)


@pytest.mark.parametrize("d", OFFSETS)
def test_lines_of_mixed_signs_at_the_bottom_of_a_binade(d):
    """lines that alternate between the two signs, and one positive value among negatives"""
    psi = np.full((2, 64, 512), -(1.0 - d) * (1 + 1j))
    psi[:, ::2] *= -1.0
    psi[:, 5, 7] = 1.0
    _check(psi)


@pytest.mark.parametrize("variant", [0, 1, 4, 5])
@pytest.mark.parametrize("n", [16, 32, 64, 128, 256, 512])
@pytest.mark.parametrize("kind", ["noise", "mode"])
def test_forward_and_backward_transforms_are_inverses(n, variant, kind):
    """With L = 0 a step is two forward / backward pairs.  Each pair rounds to FP64 once
    (0.42 u rms of the values), and its two transforms round integers whose unit is at most
    half a unit of FP64 at the line's size (0.3 u each): 0.9 u for two pairs, in quadrature.
    2 u is the bound."""
    psi = _field(kind, (16, n))
    assert _rel(_run(psi, 10.0, 0j, 0j, 1e-4, variant), psi.astype(CLD)) < 2 * U
