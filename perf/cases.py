"""Workloads of the Klein-Gordon stepper as its users run them, for timing and comparison.

A case is a plain dict.  Three kinds cover the library:

  run     one solve through the object interface (solver.Solver): initial field in, n time
          steps with the energy read at a cadence, the field and the energies out.  Real or
          complex field, Eq. (2) or the fourth-order composed scheme, the three precisions,
          device tensors or host arrays.  The library holds one context per process, so a
          pass is a whole solve; Solver is left open, as a parameter study leaves it, and
          the next solve on the same grid keeps its buffers.
  ens     a batched blow-up study (kg_ens_*): instances u0 = A exp(-|x|^2/s^2) on 64^3 and
          128^3, stepped with the threshold test, flags, levels, features and some fields out.
  train   epochs of the ranker network's training on host arrays; parameters out.
  rank    the ranker network on a sweep of points; probabilities and log times out.
"""
import math

import numpy as np
import torch

from paper_1501_04552_gb300 import kg
from paper_1501_04552_gb300.solver import Solver

L_BOX = 32.0          # side of the cube in every workload of the repository
THRESHOLD = 1e3       # blow-up threshold of the ensemble workloads
L2_BYTES = 126e6      # arrays that fit here need not travel to HBM between steps

REAL = dict(kind="run", complex=False, scheme="eq2", host=False, v0=False, noise=False)


def listed():
    return [
        # the plain 64^3 solve with the energy watched at every step: launch latency
        dict(REAL, name="bump64_energy", N=64, precision="df64", steps=100, energy_every=1, dt=0.01, A=0.5, s=1.0),
        # the smallest useful grid, many short steps, with an initial velocity
        dict(REAL, name="field32", N=32, precision="df64", steps=301, energy_every=0, dt=0.01, A=0.6, s=1.7, v0=True),
        # an everyday solve from and to host arrays
        dict(REAL, name="host128", N=128, precision="df64", steps=100, energy_every=25, dt=0.01, A=0.5, s=1.3,
             host=True),
        # the paper-scale run in the default precision: the flagship
        dict(REAL, name="field512_df64", N=512, precision="df64", steps=50, energy_every=10, dt=0.005, A=0.1, s=1.0,
             noise=True),
        # the same field with FP32 transforms and FP64 state
        dict(REAL, name="field512_mixed", N=512, precision="mixed", steps=100, energy_every=50, dt=0.005, A=0.1, s=1.0,
             noise=True),
        # IEEE FP64 throughout, the anchor that other precisions are compared with
        dict(REAL, name="field256_fp64", N=256, precision="fp64", steps=20, energy_every=10, dt=0.005, A=0.1, s=1.0,
             noise=True),
        # complex field, |u|^2 u on the full spectrum
        dict(REAL, name="complex256", N=256, precision="df64", steps=40, energy_every=20, dt=0.005, A=0.1, s=1.0,
             noise=True, complex=True),
        # fourth-order composed stepping, three passes a step
        dict(REAL, name="composed256", N=256, precision="df64", steps=15, energy_every=0, dt=0.05, A=0.1, s=1.0,
             noise=True, scheme="composed4"),
        # parametric blow-up study on mixed grids
        dict(kind="ens", name="ensemble_mixed_grids", n64=48, n128=48, precision="df64", steps=100, dt=0.005),
        # a labelling run's 64^3 batch with FP32 transforms
        dict(kind="ens", name="ensemble64_fp32", n64=256, n128=0, precision="mixed", steps=60, dt=0.005),
        # the ranker's training set, a few epochs
        dict(kind="train", name="ranker_train", rows=4096, batch=256, epochs=10),
        # the ranker over its full sweep
        dict(kind="rank", name="ranker_sweep", rows=65536),
    ]


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "ens", "ens", "train", "rank"])
    if kind == "train":
        return dict(kind=kind, rows=int(2 ** rng.uniform(9, 12)), batch=rng.choice([64, 100, 256, 512]),
                    epochs=rng.randint(1, 8))
    if kind == "rank":
        return dict(kind=kind, rows=int(2 ** rng.uniform(0, 16)))
    if kind == "ens":
        total = int(2 ** rng.uniform(0, 6.5))
        n128 = rng.randint(0, total)
        return dict(kind=kind, n64=total - n128, n128=n128, precision=rng.choice(["df64", "df64", "mixed"]),
                    steps=rng.randint(5, 50), dt=rng.choice([0.005, 0.0025]))
    N = 2 ** rng.randint(4, 9)
    precision = rng.choice(["df64", "df64", "mixed", "mixed", "fp64"])
    most = {512: 12, 256: 40, 128: 100}.get(N, 300)
    steps = rng.randint(3, max(4, most // 3 if precision == "fp64" else most))
    cplx = N < 512 and rng.random() < 0.25
    scheme = "composed4" if not cplx and rng.random() < 0.25 else "eq2"
    if scheme == "composed4":
        steps = (steps + 2) // 3
    # the FP32 transforms are meant for small fields: their rounding enters with dt^2 |u|^2
    small = precision == "mixed"
    every = 0 if scheme == "composed4" else rng.choice([0, 1, 7, 10])
    return dict(kind="run", N=N, precision=precision, steps=steps, energy_every=every, complex=cplx, scheme=scheme,
                dt=rng.choice([0.002, 0.005] if small else [0.005, 0.01]),
                A=rng.uniform(0.05, 0.15) if small else rng.uniform(0.1, 0.8), s=rng.uniform(0.8, 2.0),
                host=N <= 128 and rng.random() < 0.3, v0=rng.random() < 0.3, noise=rng.random() < 0.5)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _norm2(N, half):
    """integer |m|^2 on the spectrum of an N^3 grid, kx = 0..N/2 only when half"""
    m = torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device="cuda")
    mx = torch.arange(N // 2 + 1, dtype=torch.float64, device="cuda") if half else m
    return mx[None, None, :] ** 2 + m[None, :, None] ** 2 + m[:, None, None] ** 2


def _lowpass_noise(N, g):
    h = torch.fft.rfftn(torch.randn((N, N, N), dtype=torch.float64, device="cuda", generator=g))
    h[_norm2(N, True) > 64.0] = 0.0
    return torch.fft.irfftn(h, s=(N, N, N))


def _bump(N, A, s, centre):
    x = -L_BOX / 2 + (L_BOX / N) * torch.arange(N, dtype=torch.float64, device="cuda")
    e = [torch.exp(-((x - c) / s) ** 2) for c in centre]
    return A * e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]


def _fields(case, seed):
    """(u0, v0) on the GPU: a bump near the centre, low-passed noise, a phase when complex"""
    g = _generator(seed)
    N, A, s = case["N"], case["A"], case["s"]
    r = torch.rand(5, dtype=torch.float64, device="cuda", generator=g).tolist()
    A, s = A * (0.9 + 0.1 * r[3]), s * (0.95 + 0.1 * r[4])
    u = _bump(N, A, s, [2.0 * c - 1.0 for c in r[:3]])
    if case["noise"]:
        u = u + 1e-3 * _lowpass_noise(N, g)
    v = 0.3 * _bump(N, A, 1.5 * s, [0.0, 0.5, -0.5]) if case["v0"] else None
    if case["complex"]:
        x = -L_BOX / 2 + (L_BOX / N) * torch.arange(N, dtype=torch.float64, device="cuda")
        u = u * torch.exp(1j * (0.5 / L_BOX) * x)
        v = None if v is None else 1j * v
    return u.contiguous(), None if v is None else v.contiguous()


def _ens_inputs(case, seed):
    """grids, amplitudes U[0.5, 4], widths U[0.5, 2]"""
    rng = np.random.default_rng(seed)
    n = case["n64"] + case["n128"]
    Ns = np.array([64] * case["n64"] + [128] * case["n128"], dtype=np.int32)
    return Ns, rng.uniform(0.5, 4.0, n), rng.uniform(0.5, 2.0, n)


def _shown(case):
    """the instances whose fields are read back: every eighth, and the last"""
    n = case["n64"] + case["n128"]
    return sorted(set(range(0, n, 8)) | {n - 1})


def _net(seed):
    """He-initialised parameters, W1 (6 x 128), b1, W2 (128 x 128), b2, W3 (128 x 2), b3"""
    rng = np.random.default_rng(seed)
    p = []
    for i, o in ((6, 128), (128, 128), (128, 2)):
        p += [rng.normal(0.0, math.sqrt(2.0 / i), i * o), rng.normal(0.0, 0.05, o)]
    return np.concatenate(p).astype(np.float32)


def _rows(n, seed):
    """standardised features; labels from a curved boundary; log blow-up times"""
    rng = np.random.default_rng(seed + 1)
    X = rng.standard_normal((n, 6)).astype(np.float32)
    d = X[:, 0] + 0.5 * X[:, 1] - 0.2 * X[:, 2] ** 2
    y = (d > 0.1).astype(np.float32)
    return X, y, (1.0 - 0.5 * d + 0.05 * rng.standard_normal(n)).astype(np.float32)


def prepare(case, seed):
    st = dict(case=case)
    if case["kind"] == "run":
        st["u0"], st["v0"] = _fields(case, seed)
        if case["host"]:
            st["u0"] = st["u0"].cpu().numpy()
            st["v0"] = None if st["v0"] is None else st["v0"].cpu().numpy()
    elif case["kind"] == "ens":
        st["Ns"], st["A"], st["s"] = _ens_inputs(case, seed)
    else:
        st["params"] = _net(seed)
        st["X"], st["y"], st["logt"] = _rows(case["rows"], seed)
        st["seed"] = 1 + seed % 1000
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _chunks(steps, every):
    """steps between energy reads: after `every`, 2 `every`, ... and after the last step"""
    if not every:
        return [steps]
    return [every] * (steps // every) + ([steps % every] if steps % every else [])


def run(state):
    c = state["case"]
    if c["kind"] == "run":
        s = Solver(state["u0"], L_BOX, c["dt"], v0=state["v0"], precision=c["precision"],
                   energy_every=c["energy_every"], scheme=c["scheme"])
        E = []
        for n in _chunks(c["steps"], c["energy_every"]):
            s.step(n)
            E.append(s.energy())
        return {"u": s.field(device=not c["host"]), "E": np.array(E)}
    if c["kind"] == "ens":
        kg.kg_set_options(precision=c["precision"])
        kg.kg_ens_init(state["Ns"], L_BOX, c["dt"], state["A"], state["s"])
        kg.kg_ens_run(c["steps"], THRESHOLD)
        r = kg.kg_ens_results()
        # the library keeps max|u| as a float
        return {"frozen": r["frozen"], "level": r["level"], "maxabs": r["maxabs"].astype(np.float32),
                "features": kg.kg_ens_features(), "u": [kg.kg_ens_fetch(i) for i in _shown(c)]}
    kg.kg_mlp_set_params(state["params"])
    if c["kind"] == "train":
        kg.kg_mlp_train(state["X"], state["y"], state["logt"], epochs=c["epochs"], batch=c["batch"], lr=1e-3, T=10.0,
                        seed=state["seed"])
        return {"params": kg.kg_mlp_get_params()}
    p, t = kg.kg_mlp_predict(state["X"])
    return {"p": p, "logt": t}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _step_work(N, width, modes, transforms):
    """one evaluation of the nonlinearity with its update: two 3D transforms (5/2 n log2 n
    each for real data, 5 n log2 n for complex), the cube, six FMAs a mode.  Grids whose
    arrays do not fit in L2 move what an ideal two-pass 3D transform and the update move:
    8 work-array passes and three state arrays."""
    n = float(N) ** 3
    flops = transforms * 2.5 * n * math.log2(n) + 3.0 * n * transforms / 2 + 12.0 * modes
    fits = modes * (32 + width) <= L2_BYTES
    return flops, 0.0 if fits else modes * (8.0 * width + 48.0)


def work(case):
    if case["kind"] == "run":
        N, cplx = case["N"], case["complex"]
        modes = N * N * (N if cplx else N // 2 + 1)
        f, b = _step_work(N, 8 if case["precision"] == "mixed" else 16, modes, 4 if cplx else 2)
        passes = case["steps"] * (3 if case["scheme"] == "composed4" else 1) + 1   # and the startup level
        fields = (3 if case["v0"] else 2) * (2 if cplx else 1)
        return {"bytes": passes * b + 8.0 * N ** 3 * fields, "flops": passes * f}
    if case["kind"] == "ens":
        out = {"bytes": 0.0, "flops": 0.0}
        for N, count in ((64, case["n64"]), (128, case["n128"])):
            out["flops"] += count * (case["steps"] + 1) * _step_work(N, 16, N * N * (N // 2 + 1), 2)[0]
        out["bytes"] += sum(8.0 * (64 if i < case["n64"] else 128) ** 3 for i in _shown(case))
        return out
    macs = 6 * 128 + 128 * 128 + 128 * 2
    if case["kind"] == "train":
        used = case["epochs"] * (case["rows"] // case["batch"]) * case["batch"]
        return {"bytes": 32.0 * case["rows"] + 8.0 * 17666, "flops": 6.0 * macs * used}
    return {"bytes": 32.0 * case["rows"] + 4.0 * 17666, "flops": 2.0 * macs * case["rows"]}


# ---------------------------------------------------------------------------
# the same results from torch and numpy in 64 bits
# ---------------------------------------------------------------------------
class _Plain:
    """the scheme on the GPU with torch.fft in FP64: Eq. (2), or its fourth-order composition"""

    def __init__(self, u0, v0, dt, cplx):
        self.N, self.dt, self.cplx = u0.shape[0], dt, cplx
        self.om2 = 1.0 + (2.0 * math.pi / L_BOX) ** 2 * _norm2(self.N, not cplx)
        self.a = self.fwd(u0)
        self.v = torch.zeros_like(self.a) if v0 is None else self.fwd(v0)

    def fwd(self, u):
        return torch.fft.fftn(u) if self.cplx else torch.fft.rfftn(u)

    def inv(self, a):
        return torch.fft.ifftn(a) if self.cplx else torch.fft.irfftn(a, s=(self.N,) * 3)

    def cube(self, u):
        return self.fwd((u.real ** 2 + u.imag ** 2) * u if self.cplx else u ** 3)

    def modes(self, q):
        """(h^3/N^3) sum_k w_k q_k"""
        t = q.sum()
        if not self.cplx:
            t = 2.0 * t - q[..., 0].sum() - q[..., -1].sum()
        return float(t) * (L_BOX / self.N) ** 3 / self.N ** 3

    def quartic(self, u):
        return float((u.abs() ** 4).sum()) * (L_BOX / self.N) ** 3 / 4.0

    def eq2(self, chunks):
        w = self.dt * self.dt * self.om2 / 4.0
        c, beta = (1.0 - w) / (1.0 + w), 0.5 * self.dt * self.dt / (1.0 + w)
        a, E = self.a, []
        old = c * a - self.dt * self.v + beta * self.cube(self.inv(a))
        for n in chunks:
            for _ in range(n):
                a, old = 2.0 * c * a - old + 2.0 * beta * self.cube(self.inv(a)), a
            q = 0.5 * ((a - old).abs() / self.dt) ** 2 + 0.125 * self.om2 * (a + old).abs() ** 2
            E.append(self.modes(q) - 0.5 * (self.quartic(self.inv(a)) + self.quartic(self.inv(old))))
        return self.inv(a), E

    def composed(self, steps):
        g = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
        a, p = self.a, self.v
        F = self.cube(self.inv(a))
        for _ in range(steps):
            for h in (g * self.dt, (1.0 - 2.0 * g) * self.dt, g * self.dt):
                k = 0.5 * h / (1.0 + self.om2 * h * h / 4.0)
                p = p + k * (F - self.om2 * a)
                a = a + h * p
                F = self.cube(self.inv(a))
                p = p + k * (F - self.om2 * a)
        u = self.inv(a)
        return u, [self.modes(0.5 * (p.abs() ** 2 + self.om2 * a.abs() ** 2)) - self.quartic(u)]


def _exact_ens(case, seed):
    Ns, A, s = _ens_inputs(case, seed)
    out = {"frozen": None, "level": None, "maxabs": [], "features": [], "u": []}
    shown = _shown(case)
    for i, N in enumerate(int(n) for n in Ns):
        p = _Plain(_bump(N, A[i], s[i], [0.0, 0.0, 0.0]), None, case["dt"], False)
        w = case["dt"] ** 2 * p.om2 / 4.0
        c, beta = (1.0 - w) / (1.0 + w), 0.5 * case["dt"] ** 2 / (1.0 + w)
        m2 = _norm2(N, True)
        e = 0.5 * p.om2 * p.a.abs() ** 2
        out["features"].append([p.modes(torch.where(sel, e, 0.0)) for sel in
                                (m2 == 0, (m2 > 0) & (m2 <= 1), (m2 > 1) & (m2 <= 4), (m2 > 4) & (m2 <= 16))])
        a, old, top = p.a, None, 0.0
        old = c * a + beta * p.cube(p.inv(a))
        for _ in range(case["steps"]):
            u = p.inv(a)
            top = float(u.abs().max())
            if top > THRESHOLD:
                break
            a, old = 2.0 * c * a - old + 2.0 * beta * p.cube(u), a
        out["maxabs"].append(top)
        if i in shown:
            out["u"].append(p.inv(a).cpu().numpy())
    out["maxabs"] = np.array(out["maxabs"])
    out["features"] = np.array(out["features"])
    return out


def _forward(P, X):
    W1, b1, W2, b2, W3, b3 = P
    h1 = np.maximum(X @ W1 + b1, 0.0)
    h2 = np.maximum(h1 @ W2 + b2, 0.0)
    return h1, h2, h2 @ W3 + b3


def _split(p):
    out, k = [], 0
    for shape in ((6, 128), (128,), (128, 128), (128,), (128, 2), (2,)):
        n = int(np.prod(shape))
        out.append(p[k:k + n].reshape(shape))
        k += n
    return out


def _exact_train(st, case):
    """Adam on the unrounded network in 64 bits, the batches in the order of the library's
    shuffle: Fisher-Yates over 0..n-1 each epoch, driven by one xorshift64 stream"""
    p = st["params"].astype(np.float64)
    X, y, ell = (st[k].astype(np.float64) for k in ("X", "y", "logt"))
    n, batch = len(X), min(case["batch"], len(X))
    m, v, t, logT = np.zeros_like(p), np.zeros_like(p), 0, math.log(10.0)
    s, mask = st["seed"], (1 << 64) - 1
    for _ in range(case["epochs"]):
        perm = list(range(n))
        for i in range(n - 1, 0, -1):
            s ^= (s << 13) & mask
            s ^= s >> 7
            s ^= (s << 17) & mask
            j = s % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        for b in range(0, n - batch + 1, batch):
            idx = perm[b:b + batch]
            x, yy = X[idx], y[idx]
            P = _split(p)
            h1, h2, z = _forward(P, x)
            dz = np.empty_like(z)
            dz[:, 0] = 1.0 / (1.0 + np.exp(-z[:, 0])) - yy
            dz[:, 1] = 2.0 * yy * (z[:, 1] - ell[idx]) - 2.0 * (1.0 - yy) * np.maximum(logT - z[:, 1], 0.0)
            dz /= batch
            d2 = (dz @ P[4].T) * (h2 > 0)
            d1 = (d2 @ P[2].T) * (h1 > 0)
            g = np.concatenate([a.ravel() for a in (x.T @ d1, d1.sum(0), h1.T @ d2, d2.sum(0), h2.T @ dz, dz.sum(0))])
            t += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - 1e-3 * (m / (1.0 - 0.9 ** t)) / (np.sqrt(v / (1.0 - 0.999 ** t)) + 1e-8)
    return {"params": p}


def exact(case, seed):
    if case["kind"] == "run":
        u0, v0 = _fields(case, seed)
        p = _Plain(u0, v0, case["dt"], case["complex"])
        if case["scheme"] == "composed4":
            u, E = p.composed(case["steps"])
        else:
            u, E = p.eq2(_chunks(case["steps"], case["energy_every"]))
        return {"u": u, "E": np.array(E)}
    if case["kind"] == "ens":
        return _exact_ens(case, seed)
    st = prepare(case, seed)
    if case["kind"] == "train":
        return _exact_train(st, case)
    _, _, z = _forward(_split(st["params"].astype(np.float64)), st["X"].astype(np.float64))
    return {"p": 1.0 / (1.0 + np.exp(-z[:, 0])), "logt": z[:, 1]}
