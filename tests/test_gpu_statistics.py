"""The stopping statistics' reductions against FP64 on the host: ordinary, tiny and huge data (FP32 products
would underflow or overflow: those sums are formed in FP64), zero maps, and pixels on either side of the
violation threshold by less than FP32 resolves (counts are exact)."""
import numpy as np
import pytest

from oracle import wavelets as wav
from paper_1801_02417_gb300 import binding as B
from paper_1801_02417_gb300 import inputs
from paper_1801_02417_gb300.solver import PolarizedSARA

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1801_02417_gb300 import _build
    _build.build_library()
    B.lib()


def _violations(S, zeta):
    I, Q, U, V = S.astype(np.float64)
    p = -I + np.sqrt(Q * Q + U * U + V * V)
    return int((p > zeta).sum()), int((p > 0).sum())


@pytest.mark.parametrize("n,scale", [(16, 1.0), (64, 1.0), (64, 1e-22), (64, 1e17), (64, 0.0), (256, 1.0)])
def test_statistics_match_host(n, scale):
    rng = np.random.default_rng(n)
    M, levels = 500, 2
    uv = inputs.random_uv(M, 3, 0.5)
    S = rng.normal(size=(4, n, n))
    S[0] = np.sqrt((S[1:] ** 2).sum(0)) * (1 + rng.choice([-1e-7, 0, 1e-7, 0.3], size=(n, n)))   # on the cone's boundary
    S = (scale * S).astype(np.float32)
    Y = (scale * (rng.normal(size=(M, 4)) + 1j * rng.normal(size=(M, 4)))).astype(np.complex64)
    with PolarizedSARA(n, levels) as s:
        s.set_measurements(uv, Y if scale else np.zeros((M, 4), np.complex64), None, [0, 200, M], [1.0, 1.0])
        s.set_sara_weights(None, 0.5)
        s.set_state({"S": S})
        st = s.stats(2.0)
        coef = np.empty((4, 9, n, n), np.float32)
        B.ps_apply_psi_adjoint(s.h, S, coef)
    want = 0.5 * np.abs(coef.astype(np.float64)).sum()
    assert abs(st["weighted_l1"] - want) <= 1e-9 * want
    assert (st["violations"], st["violations_raw"]) == _violations(S, st["zeta"])
    assert (st["zeta"] > 0) == (scale > 0)
    ref = wav.psi_adjoint(S.astype(np.float64), levels)
    assert abs(st["weighted_l1"] - 0.5 * np.abs(ref).sum()) <= 1e-6 * max(np.abs(ref).sum(), 1e-300)
