"""phi^dagger of dense coverages (thousands of rows in one uv cell), where the rounding of the accumulator's FP32 sums is what
is left: every kernel width against the same interpolation in FP64.

The bound: a cell of the accumulator adds up, one after another, the runs of rows of W^2 cells, nine runs each
(W = 9: five). An FP32 addition is off by 2.5e-8 of its sum (root mean square: half an ulp evenly spread, over
the sum's binade); over n additions of random signs the errors of the growing partial sums come to 2.5e-8 sqrt(n / 2) of the
last. The weights, the transforms and the rows' own products are 1.5e-7 (a sparse coverage shows them alone). Mean of
four data sets."""
import numpy as np
import pytest

from paper_1801_02417_gb300 import binding as B
from paper_1801_02417_gb300.solver import PolarizedSARA
from problems import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1801_02417_gb300 import _build
    _build.build_library()
    B.lib()


def _adjoint64(n, uv, w, Y, W):
    K, beta = 2 * n, 2.3 * W

    def es(t):
        z = 1 - (2 * t / W) ** 2
        return np.where(z > 0, np.exp(beta * (np.sqrt(np.maximum(z, 0)) - 1)), 0.0)
    k = uv * K / (2 * np.pi)
    tap = np.floor(k + 0.5)[:, :, None] + np.arange(W) - W // 2
    wt, ix = es(tap - k[:, :, None]), tap.astype(int) % K
    cell = (ix[:, 1, :, None] * K + ix[:, 0, None, :]).ravel()
    kern = wt[:, 1, :, None] * wt[:, 0, None, :]
    rr, rl, lr, ll = (Y.astype(np.complex128) * w.astype(np.float64)[:, None]).T
    t, g = np.polynomial.legendre.leggauss(400)
    x = np.arange(n) - n // 2
    ft = (W / 2) * (np.cos(2 * np.pi / K * np.outer(x, t * W / 2)) * (g * es(t * W / 2))).sum(1)
    out = []
    for v in (rr + ll, rr - ll, rl + lr, 1j * (lr - rl)):
        a = [np.bincount(cell, weights=(c[:, None, None] * kern).ravel(), minlength=K * K) for c in (v.real, v.imag)]
        img = np.fft.ifft2((a[0] + 1j * a[1]).reshape(K, K), norm="forward").real
        out.append(img[np.ix_(x % K, x % K)] / np.outer(ft, ft))
    return np.stack(out)


@pytest.mark.parametrize("width", [5, 7, 9])
@pytest.mark.parametrize("n,M", [(32, 200001), (32, 25153), (64, 200001)])
def test_dense_cells_keep_fp32_accuracy(n, M, width):
    err = []
    for seed in range(4):
        rng = np.random.default_rng(seed)
        uv = rng.uniform(-0.4, 0.4, size=(M, 2))
        w = rng.uniform(0.7, 1.3, size=M).astype(np.float32)
        Y = (rng.normal(size=(M, 4)) + 1j * rng.normal(size=(M, 4))).astype(np.complex64)
        with PolarizedSARA(n, 2, kernel_width=width) as s:
            s.set_measurements(uv, Y, w, np.array([0, M], np.int64), np.ones(1))
            img = np.empty((4, n, n), np.float32)
            B.ps_apply_phi_adjoint(s.h, Y, img)
        err.append(rel_err(img, _adjoint64(n, uv, w, Y, width)))
    additions = width ** 2 * (5 if width == 9 else 9)
    assert np.mean(err) <= np.hypot(2.5e-8 * np.sqrt(additions / 2), 1.5e-7), err


@pytest.mark.parametrize("width", [5, 7, 9])
@pytest.mark.parametrize("M,spread", [(700, 0.1), (4097, 0.6), (4097, 1.4)])
def test_merged_blocks_at_the_wrap(M, spread, width):
    """Hundreds of rows per cell at the corner of a full grid: merged blocks whose stencils wrap in both directions, a
    last CTA with warps without rows, one cell over all warps and cells that end within a CTA. The operators'
    FP32 bound."""
    n = 32
    rng = np.random.default_rng(M + width)
    centre = np.array([31.0, -31.0])
    uv = (centre + rng.uniform(-spread, spread, size=(M, 2)) / 2) * 2 * np.pi / (2 * n)
    w = rng.uniform(0.7, 1.3, size=M).astype(np.float32)
    Y = (rng.normal(size=(M, 4)) + 1j * rng.normal(size=(M, 4))).astype(np.complex64)
    with PolarizedSARA(n, 2, kernel_width=width) as s:
        s.set_measurements(uv, Y, w, np.array([0, M], np.int64), np.ones(1))
        img = np.empty((4, n, n), np.float32)
        B.ps_apply_phi_adjoint(s.h, Y, img)
    assert rel_err(img, _adjoint64(n, uv, w, Y, width)) <= 1e-5
