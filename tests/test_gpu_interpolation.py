"""Gridding and degridding where their launch rules and splits have edges: fewer rows than a warp takes,
one more than a multiple of it, many rows in one cell (runs over several warps), one row per cell, stencils
that wrap around a full grid, and the row count and density at which a warp takes 64 rows instead of 32.

The reference is the same interpolation in FP64 (W-tap exponential-of-semicircle kernel on the 2x grid), so
what remains is FP32 rounding: the operators' FP32 bound, 1e-5 relative, for every width."""
import numpy as np
import pytest

from paper_1801_02417_gb300 import binding as B
from paper_1801_02417_gb300.solver import PolarizedSARA
from problems import rel_err

pytestmark = pytest.mark.gpu

OP_TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1801_02417_gb300 import _build
    _build.build_library()
    B.lib()


class Nufft64:
    def __init__(self, n, uv, w, W):
        self.n, self.K, self.w = n, 2 * n, w.astype(np.float64)
        beta = 2.3 * W

        def es(t):
            z = 1 - (2 * t / W) ** 2
            return np.where(z > 0, np.exp(beta * (np.sqrt(np.maximum(z, 0)) - 1)), 0.0)
        k = uv * self.K / (2 * np.pi)
        tap = np.floor(k + 0.5)[:, :, None] + np.arange(W) - W // 2
        wt = es(tap - k[:, :, None])
        ix = tap.astype(int) % self.K
        self.cell = ix[:, 1, :, None] * self.K + ix[:, 0, None, :]
        self.wt = wt[:, 1, :, None] * wt[:, 0, None, :]
        t, g = np.polynomial.legendre.leggauss(400)
        x = np.arange(n) - n // 2
        ft = (W / 2) * (np.cos(2 * np.pi / self.K * np.outer(x, t * W / 2)) * (g * es(t * W / 2))).sum(1)
        self.corr = 1.0 / np.outer(ft, ft)
        self.at = np.ix_(range(4), x % self.K, x % self.K)

    def phi(self, S):
        pad = np.zeros((4, self.K, self.K))
        pad[self.at] = S * self.corr
        G = np.fft.fft2(pad).reshape(4, -1)
        I, Q, U, V = ((G[c][self.cell] * self.wt).sum((1, 2)) * self.w for c in range(4))
        return np.stack([I + Q, U + 1j * V, U - 1j * V, I - Q], 1)

    def adjoint(self, Y):
        rr, rl, lr, ll = (Y * self.w[:, None]).T
        out = np.zeros((4, self.K * self.K), complex)
        for c, x in enumerate((rr + ll, rr - ll, rl + lr, 1j * (lr - rl))):
            np.add.at(out[c], self.cell, x[:, None, None] * self.wt)
        img = np.fft.ifft2(out.reshape(4, self.K, self.K), norm="forward").real
        return img[self.at] * self.corr


def _uv(kind, M, n):
    rng = np.random.default_rng(M + n)
    if kind == "spread":                     # the whole plane: about one row per cell, wrapped stencils
        return rng.uniform(-0.999 * np.pi, 0.999 * np.pi, size=(M, 2))
    if kind == "window":
        return rng.uniform(-0.3, 0.3, size=(M, 2))
    return np.array([0.11, -0.07]) + rng.uniform(-0.4, 0.4, size=(M, 2)) * np.pi / n   # one cell's neighbourhood


@pytest.mark.parametrize("width", [5, 7, 9])
@pytest.mark.parametrize("kind,n,M,blocks", [("spread", 16, 1, 1), ("spread", 32, 333, 5), ("spread", 64, 4001, 70),
                                             ("window", 32, 31, 1), ("window", 64, 33, 2), ("one", 32, 2000, 3),
                                             ("window", 32, 80001, 4)])
def test_phi_and_adjoint_match_fp64_interpolation(kind, n, M, blocks, width):
    uv = _uv(kind, M, n)
    rng = np.random.default_rng(7)
    w = rng.uniform(0.7, 1.3, size=M).astype(np.float32)
    S = rng.normal(size=(4, n, n)).astype(np.float32)
    Y = (rng.normal(size=(M, 4)) + 1j * rng.normal(size=(M, 4))).astype(np.complex64)
    off = np.round(np.linspace(0, M, blocks + 1)).astype(np.int64)
    with PolarizedSARA(n, 2, kernel_width=width) as s:
        s.set_measurements(uv, Y, w, off, np.full(blocks, 1.0))
        out = np.empty((M, 4), np.complex64)
        B.ps_apply_phi(s.h, S, out)
        img = np.empty((4, n, n), np.float32)
        B.ps_apply_phi_adjoint(s.h, Y, img)
        s.set_state({"S": S})
        res = s.stats()["block_residual"]
    op = Nufft64(n, uv, w, width)
    ref = op.phi(S.astype(np.float64))
    assert rel_err(out, ref) <= OP_TOL
    assert rel_err(img, op.adjoint(Y.astype(np.complex128))) <= OP_TOL
    # The per-block norms of the same rows.
    want = [np.linalg.norm(Y[off[b]:off[b + 1]] - ref[off[b]:off[b + 1]]) for b in range(blocks)]
    assert rel_err(res, np.array(want)) <= OP_TOL


# Transform lengths of every remainder modulo the stages that one pass takes, on the full grid and on a window
# of it: no stage left over, one or two, and the shortest and the longest.
@pytest.mark.parametrize("kind", ["spread", "window"])
@pytest.mark.parametrize("n", [16, 64, 128, 256, 512, 1024, 2048])
def test_every_transform_length_matches_fp64(kind, n):
    M = 60
    uv = _uv(kind, M, n)
    rng = np.random.default_rng(n)
    w = np.ones(M, np.float32)
    S = rng.normal(size=(4, n, n)).astype(np.float32)
    Y = (rng.normal(size=(M, 4)) + 1j * rng.normal(size=(M, 4))).astype(np.complex64)
    with PolarizedSARA(n, 2) as s:
        s.set_measurements(uv, Y, w, np.array([0, M], np.int64), np.ones(1))
        out = np.empty((M, 4), np.complex64)
        B.ps_apply_phi(s.h, S, out)
        img = np.empty((4, n, n), np.float32)
        B.ps_apply_phi_adjoint(s.h, Y, img)
    op = Nufft64(n, uv, w, 7)
    assert rel_err(out, op.phi(S.astype(np.float64))) <= OP_TOL
    assert rel_err(img, op.adjoint(Y.astype(np.complex128))) <= OP_TOL
