"""The SARA transforms at the edges of the launch rules: images that fit one CTA per (basis, map)
(sides up to 64, down to a coarsest side of 1), the levels of larger images handed over between
the tiled and the small kernels, and the finest level with its bases split over a cluster
(few tiles) or not. Operators against the FP64 oracle within the transforms' bound (1e-6 relative:
FP32 sums of at most 72 taps per direction), and the dual update against Algorithm 1."""
import numpy as np
import pytest

from oracle import measurement as meas
from oracle import primal_dual as opd
from oracle import wavelets as wav
from paper_1801_02417_gb300 import binding as B
from paper_1801_02417_gb300 import inputs
from paper_1801_02417_gb300.solver import PolarizedSARA
from problems import make_problem, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1801_02417_gb300 import _build
    _build.build_library()
    B.lib()


@pytest.mark.parametrize("n,levels", [(16, 1), (16, 4), (32, 3), (32, 5), (64, 1), (64, 2), (64, 6), (128, 1), (128, 2),
                                      (128, 7), (256, 3), (512, 2)])
def test_transforms_match_oracle(n, levels):
    rng = np.random.default_rng(100 + n + levels)
    S = rng.normal(size=(4, n, n)).astype(np.float32)
    A = rng.normal(size=(4, 9, n, n)).astype(np.float32)
    with PolarizedSARA(n, levels) as s:
        Sg = np.empty((4, n, n), np.float32)
        B.ps_apply_psi(s.h, A, Sg)
        Ag = np.empty((4, 9, n, n), np.float32)
        B.ps_apply_psi_adjoint(s.h, S, Ag)
    assert rel_err(Sg, wav.psi(A.astype(np.float64), levels)) <= 1e-6
    assert rel_err(Ag, wav.psi_adjoint(S.astype(np.float64), levels)) <= 1e-6


@pytest.mark.parametrize("n,levels", [(16, 4), (32, 2), (64, 6), (128, 5)])
def test_dual_update_and_reweight_match_oracle(n, levels):
    pb = make_problem(n, 300, levels, 2, seed=31)
    prob = pb["prob"]
    p = opd.step_sizes(meas.op_norm_sq_lanczos(pb["uv"], prob.w, n), opd.POLARIZED)
    st = inputs.random_state(n, 300, 33, 0.05)
    st32 = {k: (v.astype(np.complex64) if k == "B" else v.astype(np.float32)) for k, v in st.items()}
    ref = {k: v.astype(np.complex128 if k == "B" else np.float64) for k, v in st32.items()}
    W = np.random.default_rng(34).uniform(0.2, 1.0, size=(4, 9, n, n)).astype(np.float32)
    with PolarizedSARA(n, levels, tau=p.tau, rho1=p.rho1, rho2=p.rho2, rho3=p.rho3) as s:
        s.set_measurements(pb["uv"], pb["Y"], pb["w"], pb["off"], pb["eps"])
        s.set_sara_weights(W, 0.02)
        s.set_state(st32)
        s.pd_iterate(2)
        got = s.get_state()
        s.reweight(0.01)
        T = s.get_sara_weights()
    for _ in range(2):
        ref = opd.pd_iteration(ref, prob, 0.02 * W.astype(np.float64), p, opd.POLARIZED)
    for k in ("S", "A", "B"):
        assert rel_err(got[k], ref[k]) <= 2e-5 * 2, k
    # The weights of the state that was read: gamma delta / (delta + |coefficient|).
    coef = wav.psi_adjoint(got["S"].astype(np.float64), levels)
    assert rel_err(T, 0.02 * 0.01 / (0.01 + np.abs(coef))) <= 1e-5
