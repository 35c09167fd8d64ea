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


@pytest.mark.parametrize("n,levels", [(256, 2), (512, 3), (1024, 2)])
def test_dual_update_of_tiles_and_its_bounded_wait(n, levels):
    """256^2 and 512^2: one basis per CTA, the operands of the epilogue staged beside and over its input tile; 1024^2:
    the first analysis level with its input tiles shared by four bases. One iteration without data from
    a random state, A of one map against clamp(A + rho1 Psi^dagger (2 S' - S), +-gamma W); then
    a launch whose waits give up at once is reported and the handle goes on."""
    rng = np.random.default_rng(41)
    st = {k: (0.05 * rng.normal(size=s)).astype(np.float32)
          for k, s in (("S", (4, n, n)), ("Z", (2, n, n)), ("A", (4, 9, n, n)), ("C", (4, n, n)), ("D", (2, n, n)))}
    with PolarizedSARA(n, levels, tau=0.3, rho1=0.8, rho2=1.0, rho3=0.9) as s:
        s.set_measurements(np.zeros((0, 2)), np.zeros((0, 4), np.complex64), None, np.zeros(1, np.int64), np.zeros(0))
        s.set_sara_weights(None, 0.06)
        s.set_state(st)
        s.pd_iterate(1)
        got = s.get_state()
        try:
            B.ps_debug_set_wait_polls(0)
            s.pd_iterate(1)
            with pytest.raises(B.PolsaraError) as e:
                s.synchronize()
            assert e.value.status == B.PS_ETIMEOUT
        finally:
            B.ps_debug_set_wait_polls(-1)
        s.set_state(st)
        s.pd_iterate(1)
        again = s.get_state()
    X = 2 * got["S"][2:3].astype(np.float64) - st["S"][2:3]
    want = np.clip(st["A"][2:3] + 0.8 * wav.psi_adjoint(X, levels), -0.06, 0.06)
    assert rel_err(got["A"][2:3], want) <= 2e-5
    for k in ("S", "A", "C"):
        assert np.array_equal(got[k], again[k]), k
