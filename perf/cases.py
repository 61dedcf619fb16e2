"""Timed workloads of the R-SLB library, through the entry points a user calls.

Every case is one of six kinds of use:

  tube      a single shock tube (Sod): restore a checkpoint that lies on the
            device, advance it by some RK3 steps, read the populations back
            into device memory;
  fields    the 14 macroscopic output fields of a tube (Sod.moments);
  sweep     many independent tubes advanced as one batch (SodBatch), then the
            output fields of every tube;
  bjorken   many boost-invariant runs advanced as one batch (Bjorken), then
            their populations (FP64: the observables too);
  closure   a low-order tube advanced with the learned closure (closure_step);
  train     one epoch of Adam on the closure network (MLP.train).

Sizes and options are those of the repository's benchmark configurations,
convergence drivers and tests.  ``exact`` computes the same outputs in FP64
with plain torch, from the definitions.
"""
import functools
import math

import numpy as np
import torch

from paper_1612_01287_gb300 import MLP, Bjorken, Sod, SodBatch, closure_step, load

HBARC = 0.1973269804  # GeV fm
LEFT, RIGHT = (1.0, 1.0, 0.0), (0.125, 0.8, 0.0)  # chambers (n, T, beta)


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the paper-sized tube: 256 cells x 60 velocities, FP64, advanced in
        # short bursts between outputs -- latency and launches count
        dict(name="tube_256x60_f64", kind="tube", Z=256, Q_xi=20, Q_L=3, precision="f64",
             bc="outflow", tau_mode="const", tau=1e-3, steps=32),
        # a mid-sized tube with a cell count that fits no tile, fixed-equilibrium
        # ghosts and the eta/s relaxation law, as the convergence study uses
        dict(name="tube_10007x150_f32_etas", kind="tube", Z=10007, Q_xi=50, Q_L=3,
             precision="f32", bc="fixed_eq", tau_mode="etas", tau=0.3854 * 0.083, steps=16),
        # the shock tube at scale, FP32: the headline workload
        dict(name="tube_65536x600_f32", kind="tube", Z=65536, Q_xi=200, Q_L=3, precision="f32",
             bc="outflow", tau_mode="const", tau=1e-2, steps=8),
        # the same tube in FP64, the accuracy reference of the FP32 runs
        dict(name="tube_65536x600_f64", kind="tube", Z=65536, Q_xi=200, Q_L=3, precision="f64",
             bc="outflow", tau_mode="const", tau=1e-2, steps=2),
        # writing the macroscopic fields of the large tube
        dict(name="fields_65536x600_f32", kind="fields", Z=65536, Q_xi=200, Q_L=3,
             precision="f32"),
        # parameter sweep: tubes of uneven size, velocity set and relaxation time
        dict(name="sweep_64_uneven_f32", kind="sweep", nruns=64, shape_seed=4, z_lo=256,
             z_hi=8192, qxis="8,20,50,100,200", Q_L=3, precision="f32", bc="outflow",
             tau_mode="const", tau_lo=1e-4, tau_hi=10.0, steps=16),
        # convergence study in the quadrature order: equal tubes, Q_L = 2, FP64
        dict(name="sweep_16_qxi_f64", kind="sweep", nruns=16, shape_seed=0, z_lo=1000, z_hi=1000,
             qxis="4,5,6,8,10,12,16,20,30,50,70,100,150,200,300,500", Q_L=2, precision="f64",
             bc="fixed_eq", tau_mode="etas", tau_lo=0.3854 * 1e-3, tau_hi=0.3854 * 100.0,
             steps=8),
        # heavy-ion parameter scan: 16384 runs, every Q_xi from 8 to 512
        dict(name="bjorken_16384_tc", kind="bjorken", nruns=16384, shape_seed=1, q_lo=8, q_hi=512,
             Q_L=3, precision="f32", kp_mode="tf32x3", gas="parton", steps=64),
        # a small scan of the same kind: few runs per Q_xi, latency counts
        dict(name="bjorken_48_tc", kind="bjorken", nruns=48, shape_seed=2, q_lo=8, q_hi=512,
             Q_L=3, precision="f32", kp_mode="tf32x3", gas="parton", steps=64),
        # convergence study in the quadrature order, FP64 on the CUDA cores
        dict(name="bjorken_112_f64", kind="bjorken", nruns=112, shape_seed=3, q_lo=3, q_hi=100,
             Q_L=2, precision="f64", kp_mode="simt", gas="ideal", steps=50),
        # the low-order tube with the learned closure applied after every step
        dict(name="closure_65536x24", kind="closure", Z=65536, Q_xi=8, Q_L=3, hidden=64, tau=0.1,
             steps=8),
        # training the closure network: one epoch of minibatches of 8192
        dict(name="train_131072x73_h64", kind="train", n=131072, Q_xi=8, Q_L=3, hidden=64,
             batch=8192),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["tube", "tube", "tube", "fields", "sweep", "sweep", "bjorken", "bjorken",
                       "closure", "train"])
    if kind == "tube":
        f64 = rng.random() < 0.35
        mode = rng.choice(["const", "const", "etas", "none"])
        Q, QL = int(_log(rng, 4, 300)), rng.choice([2, 3, 3])
        Z = int(_log(rng, 64, 65536))
        while Z * Q * QL > (4e6 if f64 else 4e7):
            Z //= 2
        return dict(kind=kind, Z=Z, Q_xi=Q, Q_L=QL, precision="f64" if f64 else "f32",
                    bc=rng.choice(["outflow", "fixed_eq", "periodic"]), tau_mode=mode,
                    tau=_log(rng, 1e-4, 10.0),
                    steps=max(1, min(32, int((2e7 if f64 else 3e8) / (Z * Q * QL)))))
    if kind == "fields":
        Q, QL = int(_log(rng, 4, 200)), rng.choice([2, 3])
        return dict(kind=kind, Z=int(_log(rng, 256, 65536)), Q_xi=Q, Q_L=QL,
                    precision=rng.choice(["f32", "f32", "f64"]))
    if kind == "sweep":
        if rng.random() < 0.6:
            return dict(kind=kind, nruns=rng.randint(8, 64), shape_seed=rng.randrange(1 << 20),
                        z_lo=256, z_hi=8192, qxis="8,20,50,100,200", Q_L=3, precision="f32",
                        bc="outflow", tau_mode="const", tau_lo=1e-4, tau_hi=10.0,
                        steps=rng.randint(8, 16))
        Z = rng.randint(300, 1000)
        return dict(kind=kind, nruns=rng.randint(5, 16), shape_seed=0, z_lo=Z, z_hi=Z,
                    qxis="4,5,6,8,10,12,16,20,30,50,70,100,150,200,300", Q_L=2, precision="f64",
                    bc="fixed_eq", tau_mode="etas", tau_lo=0.3854 * 1e-3, tau_hi=0.3854 * 100.0,
                    steps=rng.randint(4, 8))
    if kind == "bjorken":
        if rng.random() < 0.7:
            return dict(kind=kind, nruns=int(_log(rng, 32, 8192)),
                        shape_seed=rng.randrange(1 << 20), q_lo=8, q_hi=rng.choice([128, 256, 512]),
                        Q_L=rng.choice([2, 3]), precision="f32", kp_mode="tf32x3",
                        gas=rng.choice(["parton", "ideal"]), steps=rng.randint(16, 64))
        return dict(kind=kind, nruns=int(_log(rng, 16, 128)), shape_seed=rng.randrange(1 << 20),
                    q_lo=3, q_hi=100, Q_L=2, precision="f64", kp_mode="simt",
                    gas=rng.choice(["parton", "ideal"]), steps=rng.randint(20, 50))
    if kind == "closure":
        return dict(kind=kind, Z=int(_log(rng, 512, 65536)), Q_xi=8, Q_L=3,
                    hidden=rng.choice([32, 64, 64]), tau=_log(rng, 0.05, 10.0),
                    steps=rng.randint(2, 8))
    return dict(kind=kind, n=int(_log(rng, 8192, 131072)), Q_xi=8, Q_L=3,
                hidden=rng.choice([32, 64, 64]), batch=rng.choice([2048, 4096, 8192]))


# ---------------------------------------------------------------------------
# the method in plain FP64 torch: inputs of the cases and exact outputs
# ---------------------------------------------------------------------------
def _dev(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float64), device="cuda")


def _laguerre2(Q):
    """Nodes and weights of int_0^inf e^{-x} x^2 g(x) dx."""
    i = np.arange(Q)
    x = np.linalg.eigvalsh(np.diag(2.0 * i + 3.0)
                           + np.diag(np.sqrt(i[1:] * (i[1:] + 2.0)), 1)
                           + np.diag(np.sqrt(i[1:] * (i[1:] + 2.0)), -1))

    def lag(n, t):  # L_n^{(2)} and L_{n-1}^{(2)}
        a, b = np.zeros_like(t), np.ones_like(t)
        for m in range(n):
            a, b = b, ((2.0 * m + 3.0 - t) * b - (m + 2.0) * a) / (m + 1.0)
        return b, a

    for _ in range(4):
        b, a = lag(Q, x)
        x = x - b * x / (Q * b - (Q + 2.0) * a)
    b, a = lag(Q, x)
    d = (Q * b - (Q + 2.0) * a) / x
    return x, (Q + 1.0) * (Q + 2.0) / (x * d * d)


@functools.lru_cache(maxsize=None)
def _legendre(Q):
    """Gauss-Legendre nodes and weights, the nodes polished by Newton steps."""
    x, _ = np.polynomial.legendre.leggauss(Q)

    def pq(t):
        a, b = np.zeros_like(t), np.ones_like(t)
        for m in range(Q):
            a, b = b, ((2.0 * m + 1.0) * t * b - m * a) / (m + 1.0)
        return b, a

    for _ in range(2):
        b, a = pq(x)
        x = x - b * (1.0 - x * x) / (Q * (a - x * b))
    x = 0.5 * (x - x[::-1])
    b, a = pq(x)
    d = Q * (a - x * b) / (1.0 - x * x)
    return x, 2.0 / ((1.0 - x * x) * d * d)


def _legendre_p(nm, x):
    """P_0 .. P_{nm-1} at x, stacked first."""
    p = [torch.ones_like(x), x]
    for m in range(1, nm - 1):
        p.append(((2 * m + 1) * x * p[-1] - m * p[-2]) / (m + 1))
    return torch.stack(p[:nm])


class _Set:
    """A velocity set and its f^eq expansion, FP64 on the device."""

    def __init__(self, Q, QL):
        self.Q, self.QL, self.nm = Q, QL, min(Q - 1, 5) + 1
        x, w = _legendre(Q)
        xk, wk = _laguerre2(QL)
        self.ximax = float(np.abs(x).max())
        self.x, self.w, self.xk, self.wk = _dev(x), _dev(w), _dev(xk), _dev(wk)
        self.P = _legendre_p(self.nm, self.x)  # [m][j]
        c, cw = np.polynomial.legendre.leggauss(64)
        self.c, self.cw = _dev(c), _dev(cw)
        self.Pc = _legendre_p(self.nm, self.c)

    def feq(self, n, T, beta):
        """Truncated f^eq of per-cell states: [k][j][cell]."""
        g = 1.0 / torch.sqrt((1.0 - beta) * (1.0 + beta))
        e = 1.0 / (g - g * beta * self.c[:, None])  # 1/(u0 - u c)
        X3 = (self.Pc * self.cw) @ e ** 3  # [m][cell]
        X4 = (self.Pc * self.cw) @ e ** 4
        m = torch.arange(self.nm, device="cuda", dtype=torch.float64)[:, None]
        out = []
        for k in range(self.QL):
            coef = (m + 0.5) * 0.25 * n * (X3 + (3.0 - self.xk[k]) * (X3 - T * X4))
            out.append(self.wk[k] * self.w[:, None] * (self.P.T @ coef))
        return torch.stack(out)

    def landau(self, f):
        """n, T, beta, gamma of populations f [k][j][cell]."""
        a0, a1 = f.sum(1), torch.einsum("kjs,j->ks", f, self.x)
        a2 = torch.einsum("kjs,j->ks", f, self.x * self.x)
        Nt, Nz = a0.sum(0), a1.sum(0)
        Ttt, Ttz, Tzz = self.xk @ a0, self.xk @ a1, self.xk @ a2
        Ap, Am = Ttt + 2 * Ttz + Tzz, Ttt - 2 * Ttz + Tzz
        a, b = torch.sqrt(Ap), torch.sqrt(Am)
        E = 0.5 * (Ttt - Tzz + a * b)
        beta = (a - b) / (a + b)
        g = (a + b) / (2.0 * torch.sqrt(a * b))
        n = g * (Nt - beta * Nz)
        return dict(n=n, E=E, P=E / 3, T=E / (3 * n), beta=beta, gamma=g, Nt=Nt, Nz=Nz, Ttt=Ttt,
                    Ttz=Ttz, Tzz=Tzz)

    def fields(self, f):
        """The 14 output fields, [14][cell]."""
        o = self.landau(f)
        n, T, E = o["n"], o["T"], o["E"]
        q = -4.0 * T * (o["Nz"] - n * o["beta"] * o["gamma"])
        Pi = 2.0 * E / 3.0 - (o["Ttt"] - o["Tzz"])
        return torch.stack([n, E, E / 3, T, o["beta"], o["gamma"], n / T ** 3, q, Pi, o["Nt"],
                            o["Nz"], o["Ttt"], o["Ttz"], o["Tzz"]])


def _weno(a, b, c, d, e):
    """WENO5 face flux from five upwind-ordered values (no epsilon; vanishing
    smoothness indicators by the limit of the weights)."""
    s1 = 13.0 / 12.0 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
    s2 = 13.0 / 12.0 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
    s3 = 13.0 / 12.0 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
    top = torch.maximum(s1, torch.maximum(s2, s3)).clamp_min(1e-300)
    s1, s2, s3 = (s1 / top) ** 2, (s2 / top) ** 2, (s3 / top) ** 2
    w1, w2, w3 = 0.1 * s2 * s3, 0.6 * s1 * s3, 0.3 * s1 * s2
    den = w1 + w2 + w3
    g = w1 * (2 * a - 7 * b + 5 * c) + w2 * (2 * d - b - c) + w3 * (5 * d - 4 * c - e)
    return c + torch.where(den > 1e-290, g / den, torch.zeros_like(g)) / 6.0


class _Tube:
    """One shock tube in FP64: L_Sod and its RK3 steps on f [k][j][cell]."""

    def __init__(self, vs, Z, dz, dt, bc, tau_mode, tau, left=LEFT, right=RIGHT):
        self.vs, self.Z, self.dz, self.dt, self.bc = vs, Z, dz, dt, bc
        self.tau_mode, self.tau = tau_mode, tau
        self.ghost = [vs.feq(*(_dev([v]) for v in s)) for s in (left, right)]

    def L(self, f):
        vs, x = self.vs, self.vs.x
        g = 4
        if self.bc == "periodic":
            i = torch.arange(-g, self.Z + g, device="cuda") % self.Z
            p = f[:, :, i]
        elif self.bc == "outflow":
            i = torch.arange(-g, self.Z + g, device="cuda").clamp(0, self.Z - 1)
            p = f[:, :, i]
        else:
            p = torch.cat([self.ghost[0].expand(-1, -1, g), f, self.ghost[1].expand(-1, -1, g)], 2)
        out = torch.empty_like(f)
        o = vs.landau(f) if self.tau_mode != "none" else None
        if o is not None:
            feq = vs.feq(o["n"], o["T"], o["beta"])
            tau = self.tau
            if self.tau_mode == "etas":
                tau = self.tau / o["T"] * (1.0 - 0.25 * torch.log(o["n"] / o["T"] ** 3))
        for k in range(vs.QL):
            J = x[:, None] * p[k]
            # faces s - 1/2 for s = 0 .. Z, upwind on the sign of xi
            v = [J[:, g - 3 + q: g - 3 + q + self.Z + 1] for q in range(6)]
            F = torch.where(x[:, None] > 0, _weno(*v[:5]), _weno(*v[:0:-1]))
            out[k] = -(F[:, 1:] - F[:, :-1]) / self.dz
            if o is not None:
                out[k] -= o["gamma"] * (1.0 - o["beta"] * x[:, None]) / tau * (f[k] - feq[k])
        return out

    def step(self, f):
        f1 = f + self.dt * self.L(f)
        f2 = 0.75 * f + 0.25 * (f1 + self.dt * self.L(f1))
        return f / 3.0 + (2.0 / 3.0) * (f2 + self.dt * self.L(f2))


def _np_dtype(case):
    return torch.float64 if case["precision"] == "f64" else torch.float32


def _tube_setup(case):
    """(velocity set, dz, dt) of a tube on [-1, 1]: CFL 0.5, dt below tau/2."""
    vs = _Set(case["Q_xi"], case["Q_L"])
    dz = 2.0 / case["Z"]
    dt = 0.5 * dz / vs.ximax
    if case.get("tau_mode", "const") != "none":
        dt = min(dt, 0.4 * case.get("tau", 1e-2))
    return vs, dz, dt


def _tube_state(case, seed, vs, dtype):
    """Populations of a tube in mid-run: a smoothed shock tube with seeded waves,
    each velocity a little off its equilibrium; [V][Z]."""
    rng = np.random.default_rng(seed)
    Z = case["Z"]
    z = (np.arange(Z) + 0.5) / Z
    step = 1.0 / (1.0 + np.exp((z - 0.5) / 0.05))
    a, ph = rng.uniform(0.02, 0.1, size=(3, 3)), rng.uniform(0, 2 * np.pi, size=(3, 3))
    wave = [sum(a[i, q] * np.sin(2 * np.pi * (q + 1) * z + ph[i, q]) for q in range(3))
            for i in range(3)]
    n = (0.125 + 0.875 * step) * (1.0 + wave[0])
    T = (0.8 + 0.2 * step) * (1.0 + wave[1])
    f = vs.feq(_dev(n), _dev(T), _dev(wave[2]))
    aniso = 1.0 + 0.05 * math.cos(ph[0, 0]) * (3 * vs.x ** 2 - 1)[None, :, None]
    return (f * aniso).reshape(vs.Q * vs.QL, Z).to(dtype).contiguous()


def _tube(case, dt, stream):
    mode = case.get("tau_mode", "const")
    kw = dict(tau_AW0=case["tau"], tau=1.0) if mode == "etas" else dict(tau=case.get("tau", 1e-2))
    return Sod(Z=case["Z"], Q_xi=case["Q_xi"], Q_L=case["Q_L"], precision=case["precision"],
               bc=case.get("bc", "outflow"), tau_mode=mode, dt=dt, left=LEFT, right=RIGHT,
               stream=stream, **kw)


def _get_state(tube, out):
    """Populations into device memory (rslb_get_state, on_device = 1)."""
    if load().rslb_get_state(tube._h, out.data_ptr(), 1) != 0:
        raise RuntimeError(load().rslb_last_error().decode())


def _sweep_runs(case, seed):
    """Shapes from the case alone; relaxation times and chambers from the seed."""
    sh = np.random.default_rng(case["shape_seed"])
    rng = np.random.default_rng(seed)
    qs = [int(q) for q in case["qxis"].split(",")]
    runs = []
    for r in range(case["nruns"]):
        if case["tau_mode"] == "const":
            Z = int(np.exp(sh.uniform(math.log(case["z_lo"]), math.log(case["z_hi"] + 1))))
            Q = int(sh.choice(qs))
        else:
            Z, Q = case["z_lo"], qs[r % len(qs)]
        tau = math.exp(rng.uniform(math.log(case["tau_lo"]), math.log(case["tau_hi"])))
        p = dict(Z=Z, Q_xi=Q, nL=1.0, TL=1.0, nR=0.125, TR=8.0 / rng.uniform(2.0, 20.0))
        if case["tau_mode"] == "const":
            p["tau"] = tau
            p["dt"] = min(0.5 * 2.0 / Z, 0.5 * tau)
        else:
            p.update(tau_mode="etas", tau_AW0=tau, lambda_ref=1.0,
                     dt=min(0.5 * 1.0 / Z, 0.4 * tau / max(1.0, p["TR"])))
        # far more steps than any caller asks for here: every tube stays active
        p["t_end"] = 1e6 * p["dt"]
        runs.append(p)
    return runs


def _bj_runs(case, seed):
    """Q_xi of each run from the case alone; tau_AW0 and anisotropy from the seed."""
    sh = np.random.default_rng(case["shape_seed"])
    q = sh.integers(case["q_lo"], case["q_hi"] + 1, size=case["nruns"])
    rng = np.random.default_rng(seed)
    eta_s = np.exp(rng.uniform(math.log(0.01), math.log(10.0), size=len(q)))
    T0 = rng.uniform(0.3, 0.6, size=len(q))
    return q, 5.0 * HBARC * eta_s / (0.5 * T0), rng.uniform(-0.2, 0.2, size=len(q))


def _bj_state(case, q, aniso):
    """Initial populations, concatenated per run as [k][j] (host, FP64)."""
    _, wk = _laguerre2(case["Q_L"])
    quad = {int(Q): _legendre(int(Q)) for Q in np.unique(q)}
    out = []
    for Q, a in zip(q, aniso):
        x, w = quad[int(Q)]
        f = 0.25 * w * (1.0 + 0.5 * a * (3 * x * x - 1))
        out.append(np.multiply.outer(wk, f).ravel())
    f = np.concatenate(out)
    return f if case["precision"] == "f64" else f.astype(np.float32)


def _net(case, seed):
    """Parameters and normalisation of a closure network (host, FP32)."""
    V = case["Q_xi"] * case["Q_L"]
    D, H = 3 * V + 1, case["hidden"]
    rng = np.random.default_rng(seed + 77)
    th = [rng.normal(0, 1 / math.sqrt(D), H * D), 0.1 * rng.normal(size=H),
          rng.normal(0, 1 / math.sqrt(H), H * H), 0.1 * rng.normal(size=H),
          rng.normal(0, 0.3 / math.sqrt(H), V * H), 0.02 * rng.normal(size=V)]
    mu = np.concatenate([rng.uniform(0.0, 0.08, V), rng.normal(0, 1e-3, 2 * V), [-0.5]])
    isd = np.concatenate([rng.uniform(15.0, 40.0, V), rng.uniform(50.0, 500.0, 2 * V), [0.7]])
    osd = rng.uniform(1e-5, 1e-4, V)
    return (np.concatenate(th).astype(np.float32),
            tuple(a.astype(np.float32) for a in (mu, isd, osd)))


def _train_data(case, seed):
    """Feature rows and targets on the device, FP32: each target column a smooth
    function of its row."""
    V = case["Q_xi"] * case["Q_L"]
    D = 3 * V + 1
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(case["n"], D, generator=g, device="cuda")
    A = torch.randn(D, V, generator=g, device="cuda") / math.sqrt(D)
    T = torch.tanh(X @ A) + 0.1 * torch.randn(case["n"], V, generator=g, device="cuda")
    return X, T


# ---------------------------------------------------------------------------
# what a program has in hand, and one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    stream = torch.cuda.Stream()
    kind = case["kind"]
    s = dict(kind=kind, case=case, stream=stream)
    if kind in ("tube", "fields"):
        vs, _, dt = _tube_setup(case)
        s["f0"] = _tube_state(case, seed, vs, _np_dtype(case))
        s["tube"] = _tube(case, dt, stream)
        if kind == "tube":
            s["out"] = torch.empty_like(s["f0"])
        else:
            s["out"] = torch.empty(14, case["Z"], dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            s["tube"].set_state_ptr(s["f0"].data_ptr(), 1)
    elif kind == "sweep":
        # the convergence drivers take the standard tile choice; sweeps tune
        s["batch"] = SodBatch(_sweep_runs(case, seed), Q_L=case["Q_L"],
                              precision=case["precision"], bc=case["bc"],
                              z_min=-1.0 if case["tau_mode"] == "const" else -0.5,
                              z_max=1.0 if case["tau_mode"] == "const" else 0.5,
                              autotune=case["tau_mode"] == "const", stream=stream)
    elif kind == "bjorken":
        q, t0, aniso = _bj_runs(case, seed)
        s["runs"] = Bjorken(q, case["gas"], t0, Q_L=case["Q_L"], precision=case["precision"],
                            kp_mode=case["kp_mode"], dtau=1e-3, stream=stream)
        s["runs"].set_state(_bj_state(case, q, aniso))
    else:
        theta, norm = _net(case, seed)
        V = case["Q_xi"] * case["Q_L"]
        s["mlp"] = MLP(3 * V + 1, case["hidden"], V, stream=stream)
        s["mlp"].set_params(theta)
        if kind == "closure":
            s["mlp"].set_normalization(*norm)
            tcase = dict(case, precision="f32")
            vs, _, dt = _tube_setup(tcase)
            s["f0"] = _tube_state(tcase, seed, vs, torch.float32)
            s["out"] = torch.empty_like(s["f0"])
            s["tube"] = _tube(tcase, dt, stream)
        else:
            s["X"], s["T"] = _train_data(case, seed)
    torch.cuda.synchronize()
    return s


def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "tube":
        s["tube"].set_state_ptr(s["f0"].data_ptr(), 1)
        s["tube"].step(case["steps"])
        _get_state(s["tube"], s["out"])
        return s["out"]
    if kind == "fields":
        return s["tube"].moments(out=s["out"])
    if kind == "sweep":
        s["batch"].step(case["steps"])
        got = []
        for r in range(case["nruns"]):
            m = s["batch"].moments(r)
            got.append(np.stack([m[k] for k in m]))
        got = np.concatenate(got, axis=1)
        # the fields of an FP32 batch carry FP32 digits: kept in that type
        return got if case["precision"] == "f64" else got.astype(np.float32)
    if kind == "bjorken":
        s["runs"].step(case["steps"])
        if case["precision"] == "f64":
            obs = s["runs"].read()
            return [s["runs"].get_state(), np.stack([obs[k] for k in obs])]
        return s["runs"].get_state()
    if kind == "closure":
        s["tube"].set_state_ptr(s["f0"].data_ptr(), 1)
        closure_step(s["tube"], s["mlp"], case["tau"], case["steps"])
        _get_state(s["tube"], s["out"])
        return s["out"]
    s["mlp"].train(s["X"].data_ptr(), s["T"].data_ptr(), case["n"], epochs=1, batch=case["batch"],
                   lr=2e-3, seed=12)
    return s["mlp"].get_params()


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# arithmetic per (cell, velocity) and RK stage: five moment sums (10), the WENO5
# flux of one face (60), f^eq from six coefficients (12), relaxation and update (10)
STAGE_FLOPS = 92


def work(case):
    kind = case["kind"]
    es = 8 if case.get("precision", "f32") == "f64" else 4
    if kind == "tube":  # per step: the state read and written once
        cv = case["Z"] * case["Q_xi"] * case["Q_L"] * case["steps"]
        return dict(bytes=2 * es * cv, flops=3 * STAGE_FLOPS * cv)
    if kind == "fields":
        cv = case["Z"] * case["Q_xi"] * case["Q_L"]
        return dict(bytes=es * cv + 14 * 8 * case["Z"], flops=10 * cv)
    if kind == "sweep":
        runs = _sweep_runs(case, 0)
        cv = sum(r["Z"] * r["Q_xi"] for r in runs) * case["Q_L"]
        return dict(bytes=2 * es * cv * case["steps"] + 14 * 8 * sum(r["Z"] for r in runs),
                    flops=3 * STAGE_FLOPS * cv * case["steps"])
    if kind == "bjorken":  # K^P once per distinct Q_xi; the two half-size products
        q = _bj_runs(case, 0)[0].astype(np.float64)
        state, mats = case["Q_L"] * q.sum(), 0.5 * (np.unique(q) ** 2).sum()
        return dict(bytes=es * (2 * state * case["steps"] + mats),
                    flops=3 * case["steps"] * (case["Q_L"] * (q * q).sum() + 16 * state))
    V = case["Q_xi"] * case["Q_L"]
    D, H = 3 * V + 1, case["hidden"]
    macs = D * H + H * H + H * V
    if kind == "closure":
        cv = case["Z"] * V * case["steps"]
        return dict(bytes=2 * es * cv,
                    flops=3 * STAGE_FLOPS * cv + 2 * macs * case["Z"] * case["steps"])
    return dict(bytes=4 * case["n"] * (D + V),
                flops=case["n"] * (6 * macs - 2 * D * H))


# ---------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------
def _bf16(x):
    return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def _split(theta, D, H, V):
    o, out = 0, []
    for shape in ((H, D), (H,), (H, H), (H,), (V, H), (V,)):
        n = math.prod(shape)
        out.append(theta[o:o + n].reshape(shape))
        o += n
    return out


def _exact_tube(case, seed, after=None):
    vs, dz, dt = _tube_setup(case)
    mode = case.get("tau_mode", "const")
    t = _Tube(vs, case["Z"], dz, dt, case.get("bc", "outflow"), mode, case.get("tau", 1e-2))
    f = _tube_state(case, seed, vs, _np_dtype(case)).double().reshape(vs.QL, vs.Q, case["Z"])
    for _ in range(case["steps"]):
        f = t.step(f)
        if after is not None:
            f = after(vs, f)
    return f.reshape(vs.QL * vs.Q, case["Z"])


def _closure_after(case, seed):
    """The closure's correction of a state in FP64 (BF16 weights)."""
    V = case["Q_xi"] * case["Q_L"]
    D, H = 3 * V + 1, case["hidden"]
    theta, (mu, isd, osd) = _net(case, seed)
    W1, b1, W2, b2, W3, b3 = _split(_dev(theta), D, H, V)
    W1, W2, W3 = _bf16(W1), _bf16(W2), _bf16(W3)
    mu, isd, osd = _dev(mu), _dev(isd), _dev(osd)
    silu = torch.nn.functional.silu

    def after(vs, f3):
        f = f3.reshape(V, -1)
        n = f.sum(0)
        right = torch.cat([f[:, 1:], f[:, -1:]], 1)
        left = torch.cat([f[:, :1], f[:, :-1]], 1)
        lt = torch.full_like(n, math.log10(case["tau"]))[None]
        X = (torch.cat([f / n, (right - f) / n, (f - left) / n, lt]).T - mu) * isd
        y = silu(silu(X @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
        d = n * (osd * y).T  # [v][cell]
        p = vs.xk[:, None].expand(vs.QL, vs.Q).reshape(-1)
        x = vs.x.repeat(vs.QL)
        w = (vs.wk[:, None] * vs.w).reshape(-1)
        phi = torch.stack([torch.ones_like(p), p, p * x])
        d = d - w[:, None] * (phi.T @ torch.linalg.solve((phi * w) @ phi.T, phi @ d))
        lim = torch.where((f > 0) & (d < 0), 0.5 * f / (-d).clamp_min(1e-300),
                          torch.full_like(d, 1.0))
        return (f + lim.amin(0).clamp_max(1.0) * d).reshape(f3.shape)

    return after


def _exact_sweep(case, seed):
    lo, hi = (-1.0, 1.0) if case["tau_mode"] == "const" else (-0.5, 0.5)
    sets, got = {}, []
    for r in _sweep_runs(case, seed):
        vs = sets.setdefault(r["Q_xi"], _Set(r["Q_xi"], case["Q_L"]))
        dz = (hi - lo) / r["Z"]
        left, right = (r["nL"], r["TL"], 0.0), (r["nR"], r["TR"], 0.0)
        t = _Tube(vs, r["Z"], dz, r["dt"], case["bc"], case["tau_mode"],
                  r["tau"] if case["tau_mode"] == "const" else r["tau_AW0"], left, right)
        z = lo + (np.arange(r["Z"]) + 0.5) * dz
        f = vs.feq(_dev(np.where(z < 0, r["nL"], r["nR"])), _dev(np.where(z < 0, r["TL"], r["TR"])),
                   _dev(np.zeros(r["Z"])))
        f = f.to(_np_dtype(case)).double()
        for _ in range(case["steps"]):
            f = t.step(f)
        got.append(vs.fields(f))
    return torch.cat(got, 1).cpu().numpy()


def _kp(Q, x, w):
    """K^P of one Q_xi (Eq. K_leg_disc), FP64."""
    P = _legendre_p(Q + 2, x)
    m = torch.arange(1, Q, device="cuda", dtype=torch.float64)
    Pm = P[1:Q]
    c1 = torch.where(m <= Q - 3, m * (m + 1) * (m + 2) / (2 * (2 * m + 3)), torch.zeros_like(m))
    c2 = 0.5 * m * (m + 1) * (2 * m + 1) / ((2 * m - 1) * (2 * m + 3))
    c3 = 0.5 * m * (m + 1) * (m - 1) / (2 * m - 1)
    Pm2 = torch.cat([torch.zeros_like(P[:1]), P[:Q - 2]]) if Q > 1 else P[:0]
    return w[:, None] * (Pm.T @ (c1[:, None] * P[3:Q + 2] - c2[:, None] * Pm - c3[:, None] * Pm2))


def _exact_bjorken(case, seed):
    q, t0, aniso = _bj_runs(case, seed)
    QL, dtau = case["Q_L"], 1e-3
    xk, wk = (_dev(v) for v in _laguerre2(QL))
    lag = [torch.ones_like(xk), 3.0 - xk]
    for n in range(1, QL):
        lag.append(((2 * n + 3 - xk) * lag[n] - (n + 2) * lag[n - 1]) / (n + 1))
    KL = torch.zeros(QL, QL, dtype=torch.float64, device="cuda")
    for l in range(1, QL):
        KL += torch.outer(wk * lag[l], (l + 2) * lag[l - 1] - l * lag[l]) / ((l + 1) * (l + 2))
    flat = _bj_state(case, q, aniso).astype(np.float64)
    off = np.concatenate([[0], np.cumsum(QL * q)]).astype(np.int64)
    out, obs = np.empty_like(flat), np.empty((8, len(q)))
    tau_f = 1.0 + case["steps"] * dtau
    for pad in range(64, 64 + int(q.max()), 64):  # runs whose Q_xi rounds up to pad
        qs = [int(v) for v in np.unique(q) if pad - 64 < v <= pad]
        if not qs:
            continue
        sel = [np.flatnonzero(q == v) for v in qs]
        R = max(len(s) for s in sel)
        K = torch.zeros(len(qs), pad, pad, dtype=torch.float64, device="cuda")
        xi2 = torch.zeros(len(qs), pad, dtype=torch.float64, device="cuda")
        wj = torch.zeros_like(xi2)
        f = np.zeros((len(qs), pad, R, QL))
        aw, live = np.full((len(qs), R), 1.0), np.zeros((len(qs), R), dtype=bool)
        for a, (Q, s) in enumerate(zip(qs, sel)):
            x, w = (_dev(v) for v in _legendre(Q))
            K[a, :Q, :Q] = _kp(Q, x, w)
            xi2[a, :Q], wj[a, :Q] = x * x, w
            for b, r in enumerate(s):
                f[a, :Q, b] = flat[off[r]:off[r + 1]].reshape(QL, Q).T
            aw[a, :len(s)], live[a, :len(s)] = t0[s], True
        f, aw, live = _dev(f), _dev(aw), torch.as_tensor(live, device="cuda")

        def moments(g):
            return g.sum((1, 3)), torch.einsum("ajrk,k->ar", g, xk)

        def eq(g):
            N, E = moments(g)
            P = torch.where(live, E / 3.0, torch.ones_like(E))
            if case["gas"] == "parton":
                T = P ** 0.25
                return P / T, T, aw / T
            N = torch.where(live, N, torch.ones_like(N))
            T = P / N
            return N, T, aw / T * (1.0 - 0.25 * torch.log(N / T ** 3))

        def L(g, tau):
            n_eq, T, taw = eq(g)
            feq = 0.25 * n_eq[:, None, :, None] * (wj[:, :, None, None] * wk) * (
                1.0 + (3.0 - xk) * (1.0 - T)[:, None, :, None])
            kp = torch.bmm(K, g.reshape(len(qs), pad, R * QL)).reshape(g.shape)
            return (-g + xi2[:, :, None, None] * (g @ KL.T) + kp) / tau - (
                g - feq) / taw[:, None, :, None] * live[:, None, :, None]

        for n in range(case["steps"]):
            tn = 1.0 + n * dtau
            f1 = f + dtau * L(f, tn)
            f2 = 0.75 * f + 0.25 * (f1 + dtau * L(f1, tn + dtau))
            f = f / 3.0 + (2.0 / 3.0) * (f2 + dtau * L(f2, tn + 0.5 * dtau))
        N, E = moments(f)
        _, T, _ = eq(f)
        PL = torch.einsum("ajrk,aj,k->ar", f, xi2, xk)
        o = torch.stack([torch.full_like(N, tau_f), N, E, E / 3, T, PL - E / 3, PL,
                         0.5 * (E - PL)]).cpu().numpy()
        g = f.cpu().numpy()
        for a, (Q, s) in enumerate(zip(qs, sel)):
            for b, r in enumerate(s):
                out[off[r]:off[r + 1]] = g[a, :Q, b].T.ravel()
                obs[:, r] = o[:, a, b]
    return [out, obs] if case["precision"] == "f64" else out


def _exact_train(case, seed):
    V = case["Q_xi"] * case["Q_L"]
    D, H, n = 3 * V + 1, case["hidden"], case["n"]
    X, T = (t.double() for t in _train_data(case, seed))
    theta = _dev(_net(case, seed)[0])
    # the documented minibatch order: Fisher-Yates driven by splitmix64
    mask, st = (1 << 64) - 1, 12 ^ 0x13198A2E03707344
    perm = list(range(n))
    for i in range(n - 1, 0, -1):
        st = (st + 0x9E3779B97F4A7C15) & mask
        z = ((st ^ (st >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        j = (z ^ (z >> 31)) % (i + 1)
        perm[i], perm[j] = perm[j], perm[i]
    perm = torch.as_tensor(perm, device="cuda")
    m, v = torch.zeros_like(theta), torch.zeros_like(theta)
    silu = torch.nn.functional.silu
    for t, i0 in enumerate(range(0, n, case["batch"]), 1):
        rows = perm[i0:i0 + case["batch"]]
        p = [(_bf16(a) if i % 2 == 0 else a).detach().requires_grad_(True)
             for i, a in enumerate(_split(theta, D, H, V))]
        y = silu(silu(X[rows] @ p[0].T + p[1]) @ p[2].T + p[3]) @ p[4].T + p[5]
        loss = ((y - T[rows]) ** 2).mean()
        g = torch.cat([a.reshape(-1) for a in torch.autograd.grad(loss, p)])
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        theta = theta - 2e-3 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return theta.cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "tube":
        return _exact_tube(case, seed)
    if kind == "fields":
        vs, _, _ = _tube_setup(case)
        f = _tube_state(case, seed, vs, _np_dtype(case)).double()
        return vs.fields(f.reshape(vs.QL, vs.Q, case["Z"]))
    if kind == "sweep":
        return _exact_sweep(case, seed)
    if kind == "bjorken":
        return _exact_bjorken(case, seed)
    if kind == "closure":
        return _exact_tube(dict(case, precision="f32"), seed, _closure_after(case, seed))
    return _exact_train(case, seed)
