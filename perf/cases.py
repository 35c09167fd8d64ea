"""The work that users of this framework have it do, as cases that can be timed and checked.

A case is one call, or one turn of a solve loop, through the public entry points (`binding`, `solver`):

  psi_static   the allocation-free synthesis S = Psi A              (ps_apply_psi_static)
  psi          the synthesis through a handle                       (ps_apply_psi)
  psi_adjoint  the SARA analysis Psi^dagger S                       (ps_apply_psi_adjoint)
  phi          predicted visibilities of a model image              (ps_apply_phi)
  phi_adjoint  the dirty image of a set of visibilities             (ps_apply_phi_adjoint)
  iterate      `iters` primal-dual iterations, then the state read  (ps_pd_iterate, ps_get_state)
  step         the same with the stopping-rule statistics, as a solve loop checks them
  batch        `iters` iterations of a batch of mixed-size problems (ps_batch_iterate)
  setup        a new problem from host arrays: handle, measurements, operator norm, dirty image

Inputs are seeded: compact polarized Gaussian components (whose visibilities have a closed form), Earth-rotation
uv tracks (or frequencies scattered over the whole plane), 30 dB of input SNR. Step sizes and thresholds are
given by the caller, so that `exact` can follow the same iteration in 64 bits (torch alone: a 10-tap NUFFT, good to 1e-10).
"""
import math

import numpy as np
import torch

from paper_1801_02417_gb300 import binding as B
from paper_1801_02417_gb300.solver import PolarizedSARA

OMEGA_MAX = 0.4387          # longest baseline, radians per pixel (7.2 Glambda at 2 micro-arcsecond pixels)
MODES = {"polarized": B.PS_POLARIZED, "no_constraint": B.PS_NO_CONSTRAINT, "nnls": B.PS_NNLS, "soc": B.PS_SOC,
         "tv": B.PS_TV, "tv_nc": B.PS_TV_NC, "l1tv": B.PS_L1TV, "l1tv_nc": B.PS_L1TV_NC}
CONSTRAINED = ("polarized", "soc", "tv", "l1tv")


def listed():
    return [
        # The smallest call: one synthesis of a 64 x 64 problem inside somebody else's memory pool; launches are all of it.
        {"name": "psi_static_64", "kind": "psi_static", "n": 64, "levels": 4},
        # The dictionary's analysis on its own, at the largest size of the batched mix.
        {"name": "psi_adjoint_512", "kind": "psi_adjoint", "n": 512, "levels": 5},
        # Visibilities of a model for a small image whose samples lie all over the uv plane (the whole spectrum is kept).
        {"name": "phi_full_128", "kind": "phi", "n": 128, "rows": 6001, "width": 7, "coverage": "full"},
        # Prediction for a large observation: the 1024 x 1024, 2,000,000-row workload.
        {"name": "phi_1024", "kind": "phi", "n": 1024, "rows": 2000000, "width": 7, "coverage": "tracks"},
        # Dirty image of the largest map from an odd number of rows.
        {"name": "phi_adjoint_2048", "kind": "phi_adjoint", "n": 2048, "rows": 700001, "width": 7, "coverage": "tracks"},
        # One check of the solve loop (20 iterations, then the stopping rule) on the two small workloads.
        {"name": "step_64", "kind": "step", "n": 64, "levels": 4, "rows": 2000, "blocks": 1, "mode": "polarized", "iters": 20},
        {"name": "step_256", "kind": "step", "n": 256, "levels": 4, "rows": 50000, "blocks": 8, "mode": "polarized", "iters": 20},
        # The headline workload: 1024 x 1024, 2,000,000 rows, 32 blocks, 6 levels.
        {"name": "iterate_1024", "kind": "iterate", "n": 1024, "levels": 6, "rows": 2000000, "blocks": 32, "mode": "polarized", "iters": 10},
        # The largest image, the direct cone dual, rows that divide by nothing.
        {"name": "soc_2048", "kind": "iterate", "n": 2048, "levels": 6, "rows": 700001, "blocks": 7, "mode": "soc", "iters": 8},
        # The TV problems of Algorithm 3.
        {"name": "l1tv_256", "kind": "iterate", "n": 256, "levels": 4, "rows": 50000, "blocks": 1, "mode": "l1tv", "iters": 20},
        # The batched mix (sizes 64 to 512, 2,000 to 200,000 rows), 16 problems advanced together.
        {"name": "batch_16", "kind": "batch", "problems": 16, "mix": 1, "iters": 20},
        # A request's admission: a new 256 x 256 problem from host arrays.
        {"name": "setup_256", "kind": "setup", "n": 256, "levels": 4, "rows": 50000, "blocks": 8},
    ]


def draw(rng):
    kind = rng.choice(["psi_static", "psi", "psi_adjoint", "phi", "phi_adjoint", "step", "step", "iterate", "iterate", "batch", "setup"])
    n = 2 ** rng.randint(5, 10)
    if kind == "psi_static":
        n = min(n, 256)
    levels = rng.randint(1, min(6, int(math.log2(n)) - 1))
    rows = int(math.exp(rng.uniform(math.log(1000), math.log(2e6 if n >= 512 else 2e5)))) | 1
    blocks = rng.choice([1, 3, 8, 32])
    if kind.startswith("psi"):
        return {"kind": kind, "n": n, "levels": levels}
    if kind.startswith("phi"):
        return {"kind": kind, "n": n, "rows": rows, "width": rng.choice([5, 7, 7, 9]), "coverage": rng.choice(["tracks", "full"])}
    if kind == "batch":
        return {"kind": "batch", "problems": rng.randint(4, 12), "mix": rng.randint(2, 10 ** 6), "iters": rng.randint(5, 12)}
    if kind == "setup":
        return {"kind": "setup", "n": min(n, 512), "levels": min(levels, 5), "rows": min(rows, 200001), "blocks": blocks}
    mode = rng.choice(list(MODES)) if kind == "iterate" else rng.choice(["polarized", "nnls", "soc"])
    return {"kind": kind, "n": n, "levels": levels, "rows": rows, "blocks": blocks, "mode": mode, "iters": rng.randint(3, 10 if n == 1024 else 20)}


# ---- inputs (torch and numpy alone)
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _components(n, seed, count=24):
    """Positions, widths (pixels) and Stokes amplitudes (count x 4) of compact components, sqrt(Q^2 + U^2 + V^2) < I."""
    g = _gen(seed)
    pos = _uniform(g, -0.35 * n, 0.35 * n, count, 2)
    sig = torch.exp(_uniform(g, math.log(1.2), math.log(max(2.0, n / 20)), count))
    amp = _uniform(g, 0.1, 1.0, count)
    frac, ang = _uniform(g, 0.0, 0.6, count), _uniform(g, 0.0, 2 * math.pi, count)
    return pos, sig, torch.stack([amp, amp * frac * torch.cos(ang), amp * frac * torch.sin(ang), 0.01 * amp], 1)


def _maps(n, seed):
    pos, sig, amp = _components(n, seed)
    x = torch.arange(n, device="cuda", dtype=torch.float64) - n // 2
    out = torch.zeros(4, n, n, device="cuda", dtype=torch.float64)
    for k in range(pos.shape[0]):
        ex = torch.exp(-(x - pos[k, 0]) ** 2 / (2 * sig[k] ** 2))
        ey = torch.exp(-(x - pos[k, 1]) ** 2 / (2 * sig[k] ** 2))
        out += amp[k][:, None, None] * (ey[:, None] * ex[None, :])
    return out.float().contiguous()


def _tracks(rows, seed, coverage):
    """rows x 2 frequencies in radians per pixel: every station pair over 12 h of Earth rotation, or all over the plane."""
    g = _gen(seed + 7)
    if coverage == "full":
        return _uniform(g, -0.9 * math.pi, 0.9 * math.pi, rows, 2)
    stations = 8 if rows < 20000 else (10 if rows < 500000 else 64)
    v = torch.randn(stations, 3, generator=g, device="cuda", dtype=torch.float64)
    v /= v.norm(dim=1, keepdim=True)
    a, b = torch.triu_indices(stations, stations, 1, device="cuda")
    base = v[b] - v[a]
    dumps = -(-rows // base.shape[0])
    hour = torch.linspace(-math.pi / 2, math.pi / 2, dumps, device="cuda", dtype=torch.float64)
    s, c, dec = torch.sin(hour)[None], torch.cos(hour)[None], math.radians(12.0)
    bx, by, bz = base[:, 0:1], base[:, 1:2], base[:, 2:3]
    u = s * bx + c * by
    w = -math.sin(dec) * c * bx + math.sin(dec) * s * by + math.cos(dec) * bz
    uv = torch.stack([u.reshape(-1), w.reshape(-1)], 1)
    keep = torch.sort(torch.randperm(uv.shape[0], generator=g, device="cuda")[:rows]).values
    uv = uv[keep]
    return (uv * (OMEGA_MAX / uv.norm(dim=1).max())).contiguous()


def _mix(stokes):
    """Stokes visibilities (rows x 4, complex) -> RR, RL, LR, LL."""
    i, q, u, v = stokes.unbind(1)
    return torch.stack([i + q, u + 1j * v, u - 1j * v, i - q], 1)


def _observation(n, rows, blocks, seed, coverage="tracks"):
    """uv (float64), weights (float32), noisy visibilities (complex64), block offsets, radii, noise sigma."""
    uv = _tracks(rows, seed, coverage)
    g = _gen(seed + 11)
    w = _uniform(g, 0.8, 1.2, rows).float()
    pos, sig, amp = _components(n, seed)
    stokes = torch.zeros(rows, 4, device="cuda", dtype=torch.complex128)
    r2 = (uv ** 2).sum(1)
    for k in range(pos.shape[0]):
        env = 2 * math.pi * sig[k] ** 2 * torch.exp(-0.5 * sig[k] ** 2 * r2)
        stokes += torch.polar(env, -(uv @ pos[k]))[:, None] * amp[k][None, :]
    clean = _mix(stokes) * w.double()[:, None]
    sigma = math.sqrt(float(clean.abs().square().mean()) * 1e-3)
    noise = torch.randn(rows, 4, 2, generator=g, device="cuda", dtype=torch.float64) * (sigma / math.sqrt(2))
    vis = (clean + torch.view_as_complex(noise)).to(torch.complex64)
    off = np.round(np.linspace(0, rows, blocks + 1)).astype(np.int64)
    dof = 8.0 * np.diff(off)
    return uv, w, vis, off, np.sqrt((dof + 2 * np.sqrt(2 * dof)) * sigma * sigma / 2), sigma


def _norm_bound(uv, w, n):
    """An upper bound of ||phi||^2: 2 n^2 times the largest weight of 3 x 3 uv cells of side 2 pi / n."""
    cell = torch.floor(uv * (n / (2 * math.pi))).long() + n // 2
    h = torch.bincount(cell[:, 1].clamp(0, n) * (n + 1) + cell[:, 0].clamp(0, n), weights=w.double() ** 2, minlength=(n + 1) ** 2)
    box = torch.nn.functional.avg_pool2d(h.reshape(1, 1, n + 1, n + 1), 3, 1, 1, count_include_pad=True) * 9
    return 2.0 * n * n * float(box.max())


def _steps(mode, L):
    """tau, rho1, rho2, rho3 of Section 4.3.3 (or of Algorithm 3) for ||phi||^2 <= L."""
    if "tv" in mode:
        beta, npsi = L / 2, 9.0 if "l1" in mode else 8.0
        r1, r3 = beta / (2 * npsi), beta / 2
        return 0.99 / (beta / 2 + r1 * npsi + (r3 if mode in CONSTRAINED else 0)), r1, 1.0 / L, r3
    d = 1.0 + (mode != "nnls") + (mode in ("polarized", "soc"))
    return 0.99 / d, 1.0, 1.0 / L, 1.0


def _tv_weights(L):
    return [2e-4 * L] * 4, [1e-4 * L] * 4


GAMMA = 1e-2                # threshold scale: 1e-2 of a component's amplitude (the library's default lies near it)


def _batch_sizes(case):
    r = np.random.default_rng(case["mix"])
    ns = r.choice([64, 128, 256, 512], size=case["problems"], p=[0.4, 0.3, 0.2, 0.1])
    return [{"n": int(n), "levels": 4, "rows": int(m), "blocks": int(b), "mode": "polarized"}
            for n, m, b in zip(ns, r.integers(2000, 200001, case["problems"]), r.choice([1, 4, 8], case["problems"]))]


def _coefficients(n, seed):
    g = _gen(seed + 3)
    a = torch.randn(4, 9, n, n, generator=g, device="cuda")
    return (a.abs() ** 3 * a.sign()).contiguous()       # a few large ones among many small, as a dictionary gives


def _handle(case, seed, tune):
    n, mode = case["n"], case["mode"]
    uv, w, vis, off, eps, _ = _observation(n, case["rows"], case["blocks"], seed)
    L = _norm_bound(uv, w, n)
    tau, r1, r2, r3 = _steps(mode, L)
    torch.cuda.synchronize()
    s = PolarizedSARA(n, case["levels"], mode=MODES[mode], tau=tau, rho1=r1, rho2=r2, rho3=r3)
    s.set_measurements(uv, vis, w, off, eps)
    if "tv" in mode:
        B.ps_set_tv_weights(s.h, *_tv_weights(L))
    else:
        s.set_sara_weights(None, GAMMA)
    if tune:
        B.ps_autotune(s.h, reps=3)
    return s


def _state_buffers(n, rows):
    f = lambda *shape: torch.zeros(*shape, device="cuda")  # noqa: E731
    return {"S": f(4, n, n), "Z": f(2, n, n), "A": f(4, 9, n, n),
            "B": torch.zeros(rows, 4, device="cuda", dtype=torch.complex64), "C": f(4, n, n), "D": f(2, n, n)}


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("psi_static", "psi", "psi_adjoint"):
        n = case["n"]
        if kind == "psi_adjoint":
            st["in"], st["out"] = _maps(n, seed), torch.zeros(4, 9, n, n, device="cuda")
        else:
            st["in"], st["out"] = _coefficients(n, seed), torch.zeros(4, n, n, device="cuda")
        if kind != "psi_static":
            st["s"] = PolarizedSARA(n, case["levels"])
    elif kind in ("phi", "phi_adjoint"):
        n, rows = case["n"], case["rows"]
        uv, w, vis, off, eps, _ = _observation(n, rows, 1, seed, case["coverage"])
        torch.cuda.synchronize()
        st["s"] = PolarizedSARA(n, 1, kernel_width=case["width"])
        st["s"].set_measurements(uv, vis, w, off, eps)
        if kind == "phi":
            st["in"], st["out"] = _maps(n, seed), torch.zeros(rows, 4, device="cuda", dtype=torch.complex64)
        else:
            st["in"], st["out"] = vis, torch.zeros(4, n, n, device="cuda")
    elif kind in ("iterate", "step"):
        st["s"] = _handle(case, seed, tune=True)
        st["out"] = _state_buffers(case["n"], case["rows"])
    elif kind == "batch":
        sizes = _batch_sizes(case)
        st["s"] = [_handle(c, seed + 100 * k, tune=False) for k, c in enumerate(sizes)]
        tuned = {}
        for c, s in zip(sizes, st["s"]):                # one tuning run per size class, as the server does
            key = (c["n"], c["rows"].bit_length())
            if key not in tuned:
                B.ps_autotune(s.h, reps=2)
                tuned[key] = B.ps_get_tuning(s.h)
            B.ps_set_tuning(s.h, tuned[key])
        st["b"] = B.ps_batch_create([s.h for s in st["s"]])
        st["owner"] = _BatchOwner(st["b"], st["s"])
        st["out"] = [{"S": torch.zeros(4, c["n"], c["n"], device="cuda"), "A": torch.zeros(4, 9, c["n"], c["n"], device="cuda")}
                     for c in sizes]
    else:
        uv, w, vis, off, _, sigma = _observation(case["n"], case["rows"], case["blocks"], seed)
        st.update(uv=uv.cpu().numpy(), w=w.cpu().numpy(), vis=vis.cpu().numpy(), off=off, sigma=sigma,
                  dirty=np.zeros((4, case["n"], case["n"]), np.float32))
    torch.cuda.synchronize()
    return st


class _BatchOwner:
    """Gives the batch back before its handles go."""

    def __init__(self, b, solvers):
        self.b, self.solvers = b, solvers

    def __del__(self):
        B.ps_batch_destroy(self.b)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "psi_static":
        B.ps_apply_psi_static(st["in"], st["out"], case["n"], case["levels"])
    elif kind == "psi":
        B.ps_apply_psi(st["s"].h, st["in"], st["out"])
    elif kind == "psi_adjoint":
        B.ps_apply_psi_adjoint(st["s"].h, st["in"], st["out"])
    elif kind == "phi":
        B.ps_apply_phi(st["s"].h, st["in"], st["out"])
    elif kind == "phi_adjoint":
        B.ps_apply_phi_adjoint(st["s"].h, st["in"], st["out"])
    elif kind == "iterate":
        st["s"].pd_iterate(case["iters"])
        B.ps_get_state(st["s"].h, st["out"])
    elif kind == "step":
        r = st["s"].pd_iterate(case["iters"], stats=True)
        B.ps_get_state(st["s"].h, st["out"])
        return {**st["out"], "block_residual": r["block_residual"].astype(np.float32),
                "rel_change": r["rel_change"].astype(np.float32), "zeta": float(r["zeta"]), "weighted_l1": float(r["weighted_l1"])}
    elif kind == "batch":
        B.ps_batch_iterate(st["b"], case["iters"])
        for s, out in zip(st["s"], st["out"]):
            B.ps_get_state(s.h, out)
    else:
        with PolarizedSARA(case["n"], case["levels"], noise_sigma=st["sigma"]) as s:
            s.set_measurements(st["uv"], st["vis"], st["w"], st["off"])
            B.ps_apply_phi_adjoint(s.h, st["vis"], st["dirty"])
            return {"opnorm_sq": float(s.params()["opnorm_sq"]), "gamma": float(s.config().gamma), "dirty": st["dirty"]}
    return st["out"]


# ---- what one pass cannot do without
def _iteration_work(c):
    """One iteration: every state array read and written once, read-only inputs once, the transforms' arithmetic."""
    n, rows, mode = c["n"], c["rows"], c["mode"]
    N, K = n * n, 2 * n
    fft = 2 * 2 * 5.0 * K * K * math.log2(K * K) / 4      # two packed complex images each way, three quarters pruned
    rowf = 2 * rows * (7 * 7 * 16.0 + 60)
    if "tv" in mode:
        return {"bytes": (400.0 + (96 if mode in CONSTRAINED else 0)) * N + 108.0 * rows, "flops": 200.0 * N + rowf + fft}
    per_pixel = 192.0 if mode == "polarized" else (160.0 if mode == "soc" else 96.0)
    sara = 0.0 if mode == "nnls" else 720.0 * N
    return {"bytes": per_pixel * N + sara + 108.0 * rows, "flops": (0 if mode == "nnls" else 2 * 1536.0 * N) + rowf + fft}


def work(case):
    kind = case["kind"]
    if kind.startswith("psi"):
        N = case["n"] ** 2
        return {"bytes": 160.0 * N, "flops": 1536.0 * N}
    if kind.startswith("phi"):
        n, rows, W = case["n"], case["rows"], case["width"]
        return {"bytes": 16.0 * n * n + 52.0 * rows, "flops": rows * (W * W * 16.0 + 30) + 5.0 * (2 * n) ** 2 * math.log2(4 * n * n) / 2}
    if kind == "setup":                                   # the host rows in once, about 30 products with phi^dagger phi
        n, rows = case["n"], case["rows"]
        return {"bytes": 30 * (32.0 * n * n + 104.0 * rows) + 56.0 * rows + 16.0 * n * n, "flops": 60 * rows * 800.0}
    if kind == "batch":
        each = [_iteration_work(c) for c in _batch_sizes(case)]
        return {k: case["iters"] * sum(w[k] for w in each) for k in ("bytes", "flops")}
    return {k: case["iters"] * v for k, v in _iteration_work(case).items()}


# ---- the same in 64 bits
class _Phi64:
    """phi and its adjoint: a 2x-oversampled NUFFT with a 10-tap exponential-of-semicircle kernel, in float64."""
    W = 10

    def __init__(self, n, uv, w):
        self.n, self.K, self.w = n, 2 * n, w.double()
        self.beta = 2.30 * self.W
        k = uv * (self.K / (2 * math.pi))
        c = torch.floor(k + 0.5)
        j = torch.arange(self.W, device="cuda", dtype=torch.float64) - self.W // 2
        tap = lambda d: c[:, d, None] + j + (k[:, d, None] > c[:, d, None]).double()  # noqa: E731
        tx, ty = tap(0), tap(1)
        self.ix, self.iy = tx.long() % self.K, ty.long() % self.K
        self.wx, self.wy = self._es(tx - k[:, 0, None]), self._es(ty - k[:, 1, None])
        node, gw = np.polynomial.legendre.leggauss(200)
        node, gw = torch.tensor(node, device="cuda") * (self.W / 2), torch.tensor(gw, device="cuda") * (self.W / 2)
        x = torch.arange(n, device="cuda", dtype=torch.float64) - n // 2
        ft = (torch.cos(2 * math.pi / self.K * x[:, None] * node[None]) * (gw * self._es(node))[None]).sum(1)
        self.corr = 1.0 / (ft[:, None] * ft[None, :])
        self.at = (torch.arange(n, device="cuda") - n // 2) % self.K
        self.chunk = 1 << 17

    def _es(self, t):
        z = 1 - (2 * t / self.W) ** 2
        return torch.where(z > 0, torch.exp(self.beta * (z.clamp(min=0).sqrt() - 1)), torch.zeros_like(z))

    def fwd(self, S):
        K = self.K
        pad = torch.zeros(4, K, K, device="cuda", dtype=torch.float64)
        pad[:, self.at[:, None], self.at[None, :]] = S * self.corr
        G = torch.view_as_real(torch.fft.fft2(pad).permute(1, 2, 0).contiguous()).reshape(K * K, 8)
        out = torch.empty(self.w.numel(), 8, device="cuda", dtype=torch.float64)
        for a in range(0, out.shape[0], self.chunk):
            b = slice(a, a + self.chunk)
            acc = torch.zeros_like(out[b])
            for q in range(self.W):
                for p in range(self.W):
                    acc += (self.wy[b, q] * self.wx[b, p])[:, None] * G[self.iy[b, q] * K + self.ix[b, p]]
            out[b] = acc
        return _mix(torch.view_as_complex(out.reshape(-1, 4, 2))) * self.w[:, None]

    def adj(self, Y):
        K = self.K
        rr, rl, lr, ll = (Y * self.w[:, None]).unbind(1)
        x = torch.view_as_real(torch.stack([rr + ll, rr - ll, rl + lr, 1j * (lr - rl)], 1)).reshape(-1, 8)
        acc = torch.zeros(K * K, 8, device="cuda", dtype=torch.float64)
        for a in range(0, x.shape[0], self.chunk):
            b = slice(a, a + self.chunk)
            for q in range(self.W):
                for p in range(self.W):
                    acc.index_add_(0, self.iy[b, q] * K + self.ix[b, p], (self.wy[b, q] * self.wx[b, p])[:, None] * x[b])
        H = torch.view_as_complex(acc.reshape(K, K, 4, 2)).permute(2, 0, 1)
        img = torch.fft.ifft2(H, norm="forward").real
        return img[:, self.at[:, None], self.at[None, :]] * self.corr

    def norm_sq(self):
        """||phi||^2 by Lanczos steps with full reorthogonalisation."""
        g = _gen(1)
        v = torch.randn(4, self.n, self.n, generator=g, device="cuda", dtype=torch.float64)
        V, al, be, last = [v / v.norm()], [], [], 0.0
        for _ in range(120):
            u = self.adj(self.fwd(V[-1]))
            al.append(float((u * V[-1]).sum()))
            for q in V:
                u = u - (u * q).sum() * q
            top = float(np.linalg.eigvalsh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))[-1])
            if abs(top - last) <= 1e-12 * top:
                break
            last = top
            be.append(float(u.norm()))
            V.append(u / be[-1])
        return top


def _daubechies(p):
    """Extremal-phase scaling filter of p vanishing moments (2p taps), by spectral factorisation."""
    y = np.roots([math.comb(p - 1 + k, k) for k in range(p - 1, -1, -1)]) if p > 1 else np.zeros(0)
    z = []
    for r in y:
        b = 1 - 2 * r
        s = np.sqrt(b * b - 1 + 0j)
        z.append(b - s if abs(b - s) < 1 else b + s)
    h = np.real(np.poly(np.concatenate([-np.ones(p), np.array(z)])))
    return h * (math.sqrt(2) / h.sum())


class _Psi64:
    """Dirac and db1 .. db8, periodic orthonormal 2D Mallat transforms, all scaled by 1/3."""

    def __init__(self, n, levels):
        self.n, self.levels = n, levels
        self.f = []
        for p in range(1, 9):
            h = _daubechies(p)
            self.f.append((h, np.array([(-1) ** j * h[len(h) - 1 - j] for j in range(len(h))])))

    @staticmethod
    def _down(x, h, dim):
        m = x.shape[dim]
        idx = torch.arange(0, m, 2, device=x.device)
        out = 0
        for j, c in enumerate(h):
            out = out + float(c) * x.index_select(dim, (idx + j) % m)
        return out

    @staticmethod
    def _up(lo, hi, h, g, dim):
        m = 2 * lo.shape[dim]
        shape = list(lo.shape)
        shape[dim] = m
        out = torch.zeros(shape, device=lo.device, dtype=lo.dtype)
        idx = torch.arange(0, m, 2, device=lo.device)
        for j in range(len(h)):
            out.index_add_(dim, (idx + j) % m, float(h[j]) * lo + float(g[j]) * hi)
        return out

    def ana(self, S):
        out = [S]
        for h, g in self.f:
            c, a = torch.zeros_like(S), S
            for lv in range(self.levels):
                k = (self.n >> lv) // 2
                lx, hx = self._down(a, h, 2), self._down(a, g, 2)
                c[:, :k, k:2 * k], c[:, k:2 * k, :k], c[:, k:2 * k, k:2 * k] = self._down(hx, h, 1), self._down(lx, g, 1), self._down(hx, g, 1)
                a = self._down(lx, h, 1)
            c[:, :a.shape[1], :a.shape[2]] = a
            out.append(c)
        return torch.stack(out, 1) / 3

    def syn(self, A):
        out = A[:, 0].clone()
        for b, (h, g) in enumerate(self.f):
            c = A[:, b + 1]
            k = self.n >> self.levels
            a = c[:, :k, :k]
            for _ in range(self.levels):
                lx = self._up(a, c[:, k:2 * k, :k], h, g, 1)
                hx = self._up(c[:, :k, k:2 * k], c[:, k:2 * k, k:2 * k], h, g, 1)
                a = self._up(lx, hx, h, g, 2)
                k *= 2
            out += a
        return out / 3


def _proj_e2(r, d):
    """Projection of (r, d) onto ||r|| <= d, over leading axis of r."""
    nr = r.norm(dim=0)
    a = torch.where(nr <= d, torch.ones_like(d), torch.where(nr <= -d, torch.zeros_like(d), 0.5 * (1 + d / nr.clamp(min=1e-300))))
    return a * r, torch.where(nr <= d, d, a * nr)


def _run64(c, seed, iters, stats=False):
    """`iters` iterations of Algorithm 1 (or 3) from the zero state."""
    n, mode = c["n"], c["mode"]
    uv, w, vis, off, eps, _ = _observation(n, c["rows"], c["blocks"], seed)
    L = _norm_bound(uv, w, n)
    tau, r1, r2, r3 = _steps(mode, L)
    phi, psi, Y, tv = _Phi64(n, uv, w), None, vis.to(torch.complex128), "tv" in mode
    z = lambda k: torch.zeros(k, n, n, device="cuda", dtype=torch.float64)  # noqa: E731
    st = {"S": z(4), "Z": z(2), "A": torch.zeros(4, 9, n, n, device="cuda", dtype=torch.float64), "B": torch.zeros_like(Y),
          "C": z(4), "D": z(2)}
    S, Z, A, Bd, C, D = (st[k] for k in "SZABCD")
    blk = torch.repeat_interleave(torch.arange(len(eps), device="cuda"), torch.tensor(np.diff(off), device="cuda"))
    epst = torch.tensor(eps, device="cuda")
    sumsq = lambda R: torch.zeros(len(eps), device="cuda", dtype=torch.float64).index_add_(0, blk, R.abs().square().sum(1))  # noqa: E731
    psiA, adj = z(4), z(4)
    if tv:
        mu, nu = (torch.tensor(v, device="cuda", dtype=torch.float64)[:, None, None] for v in _tv_weights(L))
    elif mode != "nnls":
        psi = _Psi64(n, c["levels"])
    for _ in range(iters):
        g = (-0.5 * phi.adj(Y - phi.fwd(S)) if tv else adj) + psiA + (C if mode in CONSTRAINED else 0)
        Sn = S - tau * g
        if mode not in CONSTRAINED:
            Sn[0].clamp_(min=0)
        X = 2 * Sn - S
        last = [float((Sn - S)[k].norm()) / max(float(S[k].norm()), 1e-300) for k in range(4)]
        S = Sn
        if mode in ("polarized", "tv", "l1tv"):
            Zn = Z - tau * D
            over = Zn[0] + Zn[1] > 0
            half = 0.5 * (Zn[0] - Zn[1])
            Zn = torch.stack([torch.where(over, half, Zn[0]), torch.where(over, -half, Zn[1])])
            Ct, Dt = C + r3 * X, D + r3 * (2 * Zn - Z)
            Z = Zn
            c0, d0 = Ct[0] / r3, Dt[0] / r3
            inside, half = c0 + d0 >= 0, 0.5 * (c0 - d0)
            p0, q0 = torch.where(inside, c0, half), torch.where(inside, d0, -half)
            p1, q1 = _proj_e2(Ct[1:] / r3, Dt[1] / r3)
            C = torch.cat([(Ct[0] - r3 * p0)[None], Ct[1:] - r3 * p1])
            D = torch.stack([Dt[0] - r3 * q0, Dt[1] - r3 * q1])
        elif mode == "soc":
            Ct = C + r3 * X
            p1, p0 = _proj_e2(Ct[1:] / r3, Ct[0] / r3)
            C = torch.cat([(Ct[0] - r3 * p0)[None], Ct[1:] - r3 * p1])
        if tv:
            ax = A[:, 0] + r1 * (X.roll(-1, 2) - X)
            ay = A[:, 1] + r1 * (X.roll(-1, 1) - X)
            k = (mu / torch.sqrt(ax * ax + ay * ay).clamp(min=1e-300)).clamp(max=1)
            A[:, 0], A[:, 1] = ax * k, ay * k
            psiA = (A[:, 0].roll(1, 2) - A[:, 0]) + (A[:, 1].roll(1, 1) - A[:, 1])
            if "l1" in mode:
                A[:, 2] = torch.minimum(torch.maximum(A[:, 2] + r1 * X, -nu), nu)
                psiA = psiA + A[:, 2]
            continue
        if psi is not None:
            A = (A + r1 * psi.ana(X)).clamp(-GAMMA, GAMMA)
            psiA = psi.syn(A)
        R = Bd / r2 + phi.fwd(X) - Y
        r = sumsq(R).sqrt()
        Bd = (r2 * (1 - (epst / r).clamp(max=1)))[blk][:, None] * R
        adj = phi.adj(Bd)
    out = {"S": S, "Z": Z, "A": A, "B": None if tv else Bd, "C": C, "D": D}
    if stats:
        R = Y - phi.fwd(S)
        img = phi.adj(R)[0]
        out.update(block_residual=sumsq(R).sqrt(), rel_change=torch.tensor(last, dtype=torch.float64),
                   zeta=3 * float(img.square().mean().sqrt()) / (2 * float((w.double() ** 2).sum())),
                   weighted_l1=float((GAMMA * (psi or _Psi64(n, c["levels"])).ana(S)).abs().sum()))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("psi_static", "psi"):
        return _Psi64(case["n"], case["levels"]).syn(_coefficients(case["n"], seed).double())
    if kind == "psi_adjoint":
        return _Psi64(case["n"], case["levels"]).ana(_maps(case["n"], seed).double())
    if kind in ("phi", "phi_adjoint"):
        uv, w, vis, *_ = _observation(case["n"], case["rows"], 1, seed, case["coverage"])
        op = _Phi64(case["n"], uv, w)
        return op.fwd(_maps(case["n"], seed).double()) if kind == "phi" else op.adj(vis.to(torch.complex128))
    if kind in ("iterate", "step"):
        return _run64(case, seed, case["iters"], stats=kind == "step")
    if kind == "batch":
        each = [_run64(c, seed + 100 * k, case["iters"]) for k, c in enumerate(_batch_sizes(case))]
        return [{"S": r["S"], "A": r["A"]} for r in each]
    uv, w, vis, *_ = _observation(case["n"], case["rows"], case["blocks"], seed)
    op = _Phi64(case["n"], uv, w)
    L, dirty = op.norm_sq(), op.adj(vis.to(torch.complex128))
    gamma = 1e-3 * float(_Psi64(case["n"], case["levels"]).ana(dirty).abs().max()) / L
    return {"opnorm_sq": L, "gamma": gamma, "dirty": dirty}
