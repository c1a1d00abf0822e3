"""Performance cases of the wildfire time step: the calls a user of the library makes, with their sizes.

A case is one pass through the public calls of ``paper_2604_19370_gb300.wf``:

* ``single``: one domain on a handle of ``wf_create``: its state in from pinned host arrays, ``steps``
  time steps, the state back out (a simulation's output interval, a served request's quantum);
* ``batch``: ``slots`` scenarios of one grid with winds of their own on a handle of
  ``wf_batch_create``: every state in, ``steps`` steps of every slot, every state out;
* ``run``: the same in the one pipelined call ``wf_batch_run``;
* ``noalloc``: a caller that owns its device arrays and advances them in place with
  ``wf_step_noalloc`` (no host copies, no graph).

Grids, orders, time step, winds, ignitions and fuel fields are those of the scenario configurations
(element size 100/64 m, dt = 1e-3, a 700 K ignition bump on 300 K, smoothed noise or two fuel
classes), at their own sizes and at ragged ones.
"""
import math

import numpy as np
import torch

from paper_2604_19370_gb300 import wf

H_ELEMENT = 100.0 / 64.0
DT = 1e-3
SCHEMES = {"pr": 0, "strang": 1, "explicit": 2}


def _case(name, kind, nx, ny, p, steps, prec="fp32", scheme="pr", rank=0, slots=1, ignitions=1, classes=False,
          per_substep=False):
    c = dict(kind=kind, nx=nx, ny=ny, p=p, steps=steps, prec=prec, scheme=scheme, rank=rank, slots=slots,
             ignitions=ignitions, classes=classes, per_substep=per_substep)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a latency-critical loop on a small domain whose device memory belongs to the caller
        _case("noalloc_128_p2_fp32", "noalloc", 128, 128, 2, 4),
        # the paper's own 64 x 64 verification run: FP64, wind with a rank-2 variation, 100 steps
        _case("verify_64_p2_fp64", "single", 64, 64, 2, 100, prec="fp64", rank=2),
        # a small ragged cubic domain, Strang / Crank-Nicolson
        _case("ragged_97x61_p3_strang_fp32", "single", 97, 61, 3, 25, scheme="strang", rank=2),
        # the million-DOF domain with wind variation: FP32 and FP64, and Strang / Crank-Nicolson
        _case("domain_1024_p2_fp32", "single", 1024, 1024, 2, 25, rank=2),
        _case("domain_1024_p2_fp64", "single", 1024, 1024, 2, 8, prec="fp64", rank=2),
        _case("domain_1024_p2_strang_fp32", "single", 1024, 1024, 2, 12, scheme="strang", rank=2),
        # the explicit comparator on a ragged domain
        _case("explicit_1030x777_p2_fp32", "single", 1030, 777, 2, 25, scheme="explicit"),
        # the largest single domain: cubic, two fuel classes with gaps, three ignitions
        _case("domain_4096_p3_fp32", "single", 4096, 4096, 3, 4, rank=2, ignitions=3, classes=True),
        # the 256-member ensemble, from and to host arrays in one call
        _case("ensemble_256x256_p2_fp32", "run", 256, 256, 2, 8, slots=256),
        # a quantum of served requests: cubic FP32 and cubic FP64 classes
        _case("quantum_8x512_p3_fp32", "batch", 512, 512, 3, 25, rank=2, slots=8),
        _case("quantum_8x256_p3_fp64", "batch", 256, 256, 3, 25, prec="fp64", rank=2, slots=8),
        # many small linear-element scenarios with F re-evaluated in the second substep
        _case("batch_40x131x97_p1_per_substep_fp32", "batch", 131, 97, 1, 25, rank=1, slots=40, per_substep=True),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["single", "single", "single", "batch", "run", "noalloc"])
    p = rng.choice([1, 2, 2, 3])
    prec = "fp32" if kind == "noalloc" else rng.choice(["fp32", "fp32", "fp64"])
    scheme = rng.choice(["pr", "pr", "pr", "strang", "explicit"])
    hi = {"single": 1500, "batch": 400, "run": 400, "noalloc": 500}[kind]
    nx, ny = size(24, hi), size(24, hi)
    dofs = (nx + p) * (ny + p)
    # DOF-steps of one pass: at most those of the listed cases of the same precision
    cap = 4e6 if prec == "fp64" else (2e7 if p == 3 else 3e7)
    slots = 1
    if kind in ("batch", "run"):
        slots = max(2, min(size(2, 64), int(cap / (2 * dofs))))
    steps = max(1, min(rng.choice([1, 4, 8, 25, 50]), int(cap / (dofs * slots))))
    return _case(None, kind, nx, ny, p, steps, prec=prec, scheme=scheme, rank=rng.choice([0, 1, 2, 2]), slots=slots,
                 ignitions=rng.choice([1, 1, 3]), classes=rng.random() < 0.25,
                 per_substep=scheme == "pr" and rng.random() < 0.2)


# ---- inputs --------------------------------------------------------------------------------------


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _greville(n, p, L):
    h = L / n
    t = np.concatenate([np.zeros(p), np.arange(n + 1) * h, np.full(p, L)])
    return np.array([t[i + 1:i + p + 1].mean() for i in range(n + p)])


def _blur(a, sigma):
    """Separable Gaussian blur with clamped edges along the last two axes."""
    r = int(math.ceil(3.0 * sigma))
    k = np.exp(-0.5 * (np.arange(-r, r + 1) / sigma) ** 2)
    k /= k.sum()
    for axis in (-1, -2):
        n = a.shape[axis]
        out = torch.zeros_like(a)
        idx = torch.arange(n, device=a.device)
        for j, w in enumerate(k):
            out += float(w) * a.index_select(axis, (idx + (j - r)).clamp(0, n - 1))
        a = out
    return a


def _inputs(case, seed):
    """Coefficient fields ([slots][Ny][Nx], in the case's precision, on the device), mean winds and
    wind-variation factors (None or per slot (fx, gx, fy, gy)), from the seed alone."""
    dev = _device()
    nx, ny, p, S = case["nx"], case["ny"], case["p"], case["slots"]
    Lx, Ly = H_ELEMENT * nx, H_ELEMENT * ny
    rs = np.random.RandomState(seed % (2 ** 32))
    xg, yg = _greville(nx, p, Lx), _greville(ny, p, Ly)
    dt = torch.float32 if case["prec"] == "fp32" else torch.float64
    X = torch.as_tensor(xg, device=dev)
    Y = torch.as_tensor(yg, device=dev)
    cx = rs.uniform(0.2 * Lx, 0.8 * Lx, (case["ignitions"], S))
    cy = rs.uniform(0.2 * Ly, 0.8 * Ly, (case["ignitions"], S))
    T = torch.full((S, ny + p, nx + p), 300.0, dtype=torch.float64, device=dev)
    for k in range(case["ignitions"]):
        ax = torch.exp(-(X[None, :] - torch.as_tensor(cx[k], device=dev)[:, None]) ** 2 / 18.0)
        ay = torch.exp(-(Y[None, :] - torch.as_tensor(cy[k], device=dev)[:, None]) ** 2 / 18.0)
        T = torch.maximum(T, 300.0 + 700.0 * ay[:, :, None] * ax[:, None, :])
    # one fuel field shared by the scenarios of a batch
    g = torch.Generator(device=dev)
    g.manual_seed(seed + 1)
    f = torch.rand((ny + p, nx + p), dtype=torch.float64, device=dev, generator=g)
    f = _blur(f, min(20.0, min(nx, ny) / 8.0))
    f = (f - f.min()) / (f.max() - f.min())
    if case["classes"]:
        f = torch.where(f > f.flatten().kthvalue(f.numel() // 2).values, 1.0, 0.2).to(torch.float64)
        gaps = torch.rand((ny // 8 + 1, nx // 8 + 1), device=dev, generator=g) < 0.05
        gaps = gaps.repeat_interleave(8, 0).repeat_interleave(8, 1)
        gaps = torch.nn.functional.pad(gaps, (0, 8, 0, 8))[:ny + p, :nx + p]
        f = torch.where(gaps, 0.0, f)
    fuel = f[None].expand(S, -1, -1)
    speed, angle = rs.uniform(0.0, 3.0, S), rs.uniform(0.0, 2.0 * math.pi, S)
    winds = [(float(s * math.cos(t)), float(s * math.sin(t))) for s, t in zip(speed, angle)]
    factors = None
    if case["rank"]:
        def series(x, L):
            a, ph = rs.uniform(-1.0, 1.0, 4), rs.uniform(0.0, 2.0 * math.pi, 4)
            return sum(a[m] * np.cos((m + 1) * math.pi * x / L + ph[m]) for m in range(4)) / np.abs(a).sum()

        factors = []
        for s in range(S):
            amp = 0.1 * speed[s] / case["rank"]
            factors.append(tuple(np.stack([w * series(x, L) for _ in range(case["rank"])])
                                 for w, x, L in ((amp, xg, Lx), (1.0, yg, Ly), (amp, xg, Lx), (1.0, yg, Ly))))
    return T.to(dt).contiguous(), fuel.to(dt).contiguous(), winds, factors


class State:
    """A handle with its operators built and the caller's arrays; the handle is freed with it."""

    def __init__(self, case):
        self.case = case
        self.h = None

    def __del__(self):
        if self.h:
            wf.wf_destroy(self.h)
            self.h = None


def prepare(case, seed):
    T, fuel, winds, factors = _inputs(case, seed)
    st = State(case)
    prm = wf.wf_params_default(
        Lx=H_ELEMENT * case["nx"], Ly=H_ELEMENT * case["ny"], wind_x=winds[0][0], wind_y=winds[0][1],
        precision=wf.WF_FP32 if case["prec"] == "fp32" else wf.WF_FP64, scheme=SCHEMES[case["scheme"]],
        F_timing=wf.WF_F_PER_SUBSTEP if case["per_substep"] else wf.WF_F_ONCE)
    n1 = T[0].numel()
    st.n = T.numel()
    if case["slots"] == 1:
        st.h = wf.wf_create(case["nx"], case["ny"], case["p"], DT, prm)
        if factors:
            wf.wf_set_wind(st.h, case["rank"], np.concatenate([a.ravel() for a in factors[0]]))
    else:
        st.h = wf.wf_batch_create(case["nx"], case["ny"], case["p"], DT, prm, case["slots"])
        zero = np.zeros(n1)
        for s in range(case["slots"]):
            if factors:
                wf.wf_batch_set_slot(st.h, s, zero, zero, winds[s][0], winds[s][1], case["rank"],
                                     np.concatenate([a.ravel() for a in factors[s]]))
            else:
                wf.wf_set_mean_wind(st.h, winds[s][0], winds[s][1], slot=s)
            wf.wf_batch_activate(st.h, s, True)
    if case["kind"] == "noalloc":
        st.T0, st.f0 = T[0], fuel[0]
        st.T, st.f = torch.empty_like(st.T0), torch.empty_like(st.f0)
    else:
        pin = torch.cuda.is_available()
        st.T0, st.f0, st.T, st.f = (torch.empty(T.shape, dtype=T.dtype, pin_memory=pin) for _ in range(4))
        st.T0.copy_(T)
        st.f0.copy_(fuel)
    return st


def run(st):
    c, h, n = st.case, st.h, st.n
    f32 = c["prec"] == "fp32"
    src, dst = (st.T0.data_ptr(), st.f0.data_ptr()), (st.T.data_ptr(), st.f.data_ptr())
    if c["kind"] == "noalloc":
        # on the caller's stream (1 names the legacy default stream, which torch reports as 0)
        wf.wf_set_stream(h, torch.cuda.current_stream().cuda_stream or 1)
        st.T.copy_(st.T0)
        st.f.copy_(st.f0)
        code = wf.wf_step_noalloc(h, dst[0], dst[1], c["nx"] + c["p"], c["steps"])
        if code != wf.WF_OK:
            raise wf.WFError(code, "wf_step_noalloc")
    elif c["kind"] == "run":
        wf.wf_batch_run_ptr(h, *src, *dst, n, c["steps"], min(8, c["slots"]), f32)
    elif c["kind"] == "batch":
        wf.wf_batch_states_ptr(h, *src, n, f32, True)
        wf.wf_step(h, c["steps"])
        wf.wf_batch_states_ptr(h, *dst, n, f32, False)
    else:
        (wf.wf_set_state_f32_ptr if f32 else wf.wf_set_state_ptr)(h, *src, n)
        wf.wf_step(h, c["steps"])
        (wf.wf_get_state_f32_ptr if f32 else wf.wf_get_state_ptr)(h, *dst, n)
    return [st.T, st.f]


def work(case):
    """One pass: T and fuel read and written once, and every step's sum-factorised operations: its
    quadratures (two per step for Strang and for F per substep) and line solves."""
    p = case["p"]
    q, W = p + 1, 2 * p + 1
    dofs = (case["nx"] + p) * (case["ny"] + p) * case["slots"]
    interp = 2 * q * q + 3 * q * q * q
    fuel = q * q + q * q * q
    quad = 2 * (interp + fuel) + 6 * q * q + 4 * W + 1
    quads = 2 if case["scheme"] == "strang" or case["per_substep"] else 1
    # a line solve is 4p + 1 per value; T and fuel along x and y, and for two quadratures T again
    solves = 4 + 2 * (quads - 1)
    size = 4 if case["prec"] == "fp32" else 8
    flops = 2 * (quads * quad + solves * (4 * p + 1)) * dofs * case["steps"]
    return {"bytes": 4 * size * dofs, "flops": flops}


# ---- the scheme in 64 bits -----------------------------------------------------------------------


class _Direction:
    """Open uniform B-splines of degree p on n elements: tables at the q = p+1 Gauss points of every
    element, [n][q][p+1], and the dense mass, stiffness and advection matrices."""

    def __init__(self, n, p, L, dev):
        q, h = p + 1, L / n
        x, w = np.polynomial.legendre.leggauss(q)
        xi, self.w = 0.5 * (x + 1.0), torch.as_tensor(0.5 * w * h, device=dev)
        # in units of the element size: knots are integers, clamped to [0, n]
        e = np.arange(n)
        t = lambda i: np.clip(e[:, None] + i, 0, n).astype(float)  # noqa: E731  knot i of element e
        pos = e[:, None] + xi[None, :]
        N = [np.ones((n, q))]
        low = None
        for k in range(1, p + 1):
            low, new = N, []
            for a in range(k + 1):
                v = np.zeros((n, q))
                if a > 0:
                    lo, hi = t(a - k), t(a)
                    v += (pos - lo) / (hi - lo) * N[a - 1]
                if a < k:
                    lo, hi = t(a - k + 1), t(a + 1)
                    v += (hi - pos) / (hi - lo) * N[a]
                new.append(v)
            N = new
        D = []
        for a in range(p + 1):
            v = np.zeros((n, q))
            if a > 0:
                v += p / (t(a) - t(a - p)) * low[a - 1]
            if a < p:
                v -= p / (t(a + 1) - t(a - p + 1)) * low[a]
            D.append(v / h)
        self.n, self.p, self.q, self.N = n, p, q, n + p
        self.B = torch.as_tensor(np.stack(N, -1), device=dev)
        self.D = torch.as_tensor(np.stack(D, -1), device=dev)
        self.M, self.K, self.G = (self._matrix(u, v) for u, v in ((self.B, self.B), (self.D, self.D),
                                                                 (self.B, self.D)))

    def _matrix(self, test, trial):
        A = torch.zeros((self.N, self.N), dtype=torch.float64, device=test.device)
        e = torch.arange(self.n, device=test.device)
        for a in range(self.p + 1):
            for b in range(self.p + 1):
                A.index_put_((e + a, e + b), (self.w * test[:, :, a] * trial[:, :, b]).sum(1), accumulate=True)
        return A

    def at_points(self, c, tab):
        """Spline along the last axis at the Gauss points: [..., N] -> [..., n, q]."""
        return sum(c[..., k:k + self.n, None] * tab[:, :, k] for k in range(self.p + 1))

    def against(self, v, tab):
        """Its transpose: [..., n, q] -> [..., N]."""
        out = torch.zeros(v.shape[:-2] + (self.N,), dtype=v.dtype, device=v.device)
        for k in range(self.p + 1):
            out[..., k:k + self.n] += (v * tab[:, :, k]).sum(-1)
        return out

    def band_apply(self, A, c):
        """Banded matrix (or one per slot, [S][N][N]) along the last axis of c ([S][..][N])."""
        out = torch.zeros_like(c)
        for d in range(-self.p, self.p + 1):
            lo, hi = max(0, -d), min(self.N, self.N - d)
            diag = torch.diagonal(A, d, -2, -1)
            out[..., lo:hi] += (diag[:, None, :] if A.dim() == 3 else diag) * c[..., lo + d:hi + d]
        return out


def exact(case, seed):
    dev = _device()
    T, phi, winds, factors = _inputs(case, seed)
    T, phi = T.to(torch.float64), phi.to(torch.float64)
    nx, ny, p, S = case["nx"], case["ny"], case["p"], case["slots"]
    X = _Direction(nx, p, H_ELEMENT * nx, dev)
    Y = _Direction(ny, p, H_ELEMENT * ny, dev)
    # the model constants of the default parameters, divided by rho c_p
    inv = 1.0 / 1.293
    C_d, c_W, c_chi = 0.3 * inv, 0.5, 2e-2 * inv
    C_nld, c_rad = 4.0 * 5.67e-8 * 0.05 * (3.5e-2 / 0.05) * inv, 5.67e-8 * 0.05 / (1.5 * 0.05) * inv
    K_ign, k_f = 1e4 * 1.293 * 70.0 * 1e-4 * inv, 300.0 * 1e-4
    T_a, T_amb, T_ig, phi_min = 300.0, 300.0, 800.0, 0.2 + 1e-6
    bx = torch.tensor([w[0] for w in winds], dtype=torch.float64, device=dev)[:, None, None]
    by = torch.tensor([w[1] for w in winds], dtype=torch.float64, device=dev)[:, None, None]
    Ax = C_d * X.K + c_W * bx * X.G + c_chi * X.M
    Ay = C_d * Y.K + c_W * by * Y.G
    bp = None
    if factors:
        tens = [torch.as_tensor(np.stack([f[k] for f in factors]), device=dev) for k in range(4)]
        pts = [d.at_points(t, d.B) for d, t in zip((X, Y, X, Y), tens)]  # [S][rank][n][q]
        bp = [torch.einsum("srya,srxb->syaxb", pts[k + 1], pts[k]) for k in (0, 2)]
    wt = Y.w[None, :, None, None] * X.w  # [1][qy][1][qx]

    def along_y(f, c, *args):
        return f(c.transpose(-1, -2), *args).transpose(-1, -2)

    def at_points(c, tx, ty):
        v = X.at_points(c, tx)                       # [S][Ny][nx][qx]
        return sum(v[:, l:l + ny, None] * ty[:, :, l][:, :, None, None] for l in range(p + 1))

    def against(v, tx, ty):
        u = X.against(v, tx)                          # [S][ny][qy][Nx]
        out = torch.zeros((S, Y.N, X.N), dtype=torch.float64, device=dev)
        for l in range(p + 1):
            out[:, l:l + ny] += (u * ty[:, :, l][:, :, None]).sum(2)
        return out

    def load(T, phi, with_fuel):
        """F and the load vector of the fuel increment -tau k_f E phi."""
        v = at_points(T, X.B, Y.B)
        ph = at_points(phi, X.B, Y.B)
        burn = (v > T_ig) & (ph > phi_min)
        E = torch.where(burn, v * torch.exp(-T_a / torch.where(burn, v, 1.0)), 0.0)
        G = against(wt * (-DT * k_f) * E * ph, X.B, Y.B) if with_fuel else None
        s = K_ign * E + c_chi * T_amb + c_rad * (T_amb ** 4 - v ** 4)
        q = -C_nld * v ** 3
        del v, ph, burn, E
        gx, gy = at_points(T, X.D, Y.B), at_points(T, X.B, Y.D)
        if bp is not None:
            s -= c_W * (bp[0] * gx + bp[1] * gy)
        gx *= q * wt
        gy *= q * wt
        s *= wt
        return against(s, X.B, Y.B) + against(gx, X.D, Y.B) + against(gy, X.B, Y.D), G

    iMx, iMy = torch.linalg.inv(X.M), torch.linalg.inv(Y.M)

    def solve(ix, iy, R):
        return iy @ (R @ ix.transpose(-1, -2))

    def diffuse(T):
        """(A_x (x) M^y) T and (M^x (x) A_y) T."""
        return (along_y(lambda c: Y.band_apply(Y.M, c), X.band_apply(Ax, T)),
                along_y(lambda c: Y.band_apply(Ay, c), X.band_apply(X.M, T)))

    # every system is solved for the increment of T: the same equations, less rounding
    if case["scheme"] == "pr":
        th = 0.5 * DT
        iX, iY = torch.linalg.inv(X.M + th * Ax), torch.linalg.inv(Y.M + th * Ay)
    elif case["scheme"] == "strang":
        iX, iY = torch.linalg.inv(X.M + 0.25 * DT * Ax), torch.linalg.inv(Y.M + 0.5 * DT * Ay)
    for _ in range(case["steps"]):
        F, G = load(T, phi, True)
        if case["scheme"] == "explicit":
            T1 = T + solve(iMx, iMy, DT * (F - sum(diffuse(T))))
        elif case["scheme"] == "pr":
            T1 = T + solve(iX, iMy, th * (F - sum(diffuse(T))))
            if case["per_substep"]:
                F = load(T1, phi, False)[0]
            T1 = T1 + solve(iMx, iY, th * (F - sum(diffuse(T1))))
        else:
            T1 = T + solve(iX, iMy, 0.5 * DT * (F - diffuse(T)[0]))
            T1 = T1 + iY @ (-DT * along_y(lambda c: Y.band_apply(Ay, c), T1))
            T1 = T1 + solve(iX, iMy, 0.5 * DT * (load(T1, phi, False)[0] - diffuse(T1)[0]))
        phi = phi + solve(iMx, iMy, G)
        T = T1
    if case["kind"] == "noalloc":
        return [T[0], phi[0]]
    return [T, phi]
