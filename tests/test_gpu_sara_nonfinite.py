"""An infinity or a NaN in one pixel: the coefficients whose filters reach it are not finite, and no others. (A filter
padded with zero taps would spread it, 0 x infinity being NaN.) Sizes that take every form of the analysis: all levels in
one launch, tiles of one basis and of four, and the small levels with unrolled filters and with loops."""
import numpy as np
import pytest

from oracle import wavelets as wav
from paper_1801_02417_gb300 import binding as B
from paper_1801_02417_gb300.solver import PolarizedSARA

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1801_02417_gb300 import _build
    _build.build_library()
    B.lib()


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("n,levels", [(64, 3), (128, 3), (256, 4), (1024, 2)])
def test_nonfinite_pixel_stays_within_the_filters_reach(n, levels, bad):
    rng = np.random.default_rng(n)
    S = rng.normal(size=(4, n, n)).astype(np.float32)
    S[2, n // 2 + 5, n // 3 | 1] = bad
    S[1, 0, 0] = bad
    A = np.empty((4, 9, n, n), np.float32)
    with PolarizedSARA(n, levels) as s:
        B.ps_apply_psi_adjoint(s.h, S, A)
    maps = [1, 2] if n < 1024 else [2]
    with np.errstate(invalid="ignore"):
        ref = wav.psi_adjoint(S[maps].astype(np.float64), levels)
    assert np.isfinite(A[[0, 3]]).all()
    for k, r in zip(maps, ref):
        for b in range(9):
            assert np.array_equal(np.isfinite(A[k, b]), np.isfinite(r[b])), (k, b)
            assert 0 < (~np.isfinite(r[b])).sum() < n * n
