"""The stopping statistics' FP64 sums of FP32 products, compared with the exact sums: products whose rounding error is
not zero, and sums short enough that no averaging hides a lost part of one. What a sum may be off is counted in
roundings to 53 bits: one where eight products make the whole sum, one per level of the reduction otherwise."""
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_1801_02417_gb300 import binding as B
from paper_1801_02417_gb300.solver import PolarizedSARA

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1801_02417_gb300 import _build
    _build.build_library()
    B.lib()


def _exact_dot(a, b):
    return sum((Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b)), Fraction(0))


@pytest.mark.parametrize("seed", range(8))
@pytest.mark.parametrize("spread", [1.0, 1e-3])
def test_weighted_norm_of_one_group_of_products(seed, spread):
    """Weights that are zero but for the eight coefficients that one thread adds up as a group (four of the first
    map's Dirac part and, 65,536 x 4 coefficients on, four of the second map's db7 part)."""
    n, levels = 128, 3
    rng = np.random.default_rng(seed)
    S = rng.normal(size=(4, n, n)).astype(np.float32)
    W = np.zeros((4, 9, n, n), np.float32)
    at = np.r_[0:4, 4 * 65536:4 * 65536 + 4]
    W.reshape(-1)[at] = rng.uniform(0.3, 1.0, size=8) * spread ** rng.uniform(0, 1, size=8)
    with PolarizedSARA(n, levels, gamma=1.0) as s:
        s.set_measurements(np.array([[0.1, 0.2]]), np.zeros((1, 4), np.complex64), None, [0, 1], [1.0])
        s.set_sara_weights(W, 0.7)
        s.set_state({"S": S})
        got = s.stats()["weighted_l1"]
        T = s.get_sara_weights().reshape(-1)[at]
        coef = np.empty((4, 9, n, n), np.float32)
        B.ps_apply_psi_adjoint(s.h, S, coef)
    want = _exact_dot(T, np.abs(coef.reshape(-1)[at]))
    assert want > 0
    assert abs(Fraction(got) - want) <= want * Fraction(1, 2 ** 52)


@pytest.mark.parametrize("n", [16, 64, 128])
def test_residual_rms_of_one_visibility(n):
    """zeta of a zero image is that of the dirty image, which one row makes the same on every run. Sum of squares: 13
    additions in a CTA and 13 over the CTAs, two more for a thread's groups (128^2 and below), then the root."""
    rng = np.random.default_rng(n)
    Y = (rng.normal(size=(1, 4)) + 1j * rng.normal(size=(1, 4))).astype(np.complex64)
    w = np.array([0.83], np.float32)
    with PolarizedSARA(n, 2) as s:
        s.set_measurements(np.array([[0.31, -0.17]]), Y, w, [0, 1], [1.0])
        s.set_state({"S": np.zeros((4, n, n), np.float32)})
        got = s.stats(2.0)["zeta"]
        dirty = np.empty((4, n, n), np.float32)
        B.ps_apply_phi_adjoint(s.h, Y, dirty)
    q = float(_exact_dot(dirty[0].reshape(-1), dirty[0].reshape(-1)))
    want = 2.0 * math.sqrt(q / n ** 2) / (2.0 * float(w[0]) ** 2)
    assert abs(got - want) <= 32 * 2.0 ** -53 * want
