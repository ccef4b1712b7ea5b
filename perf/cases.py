"""The work that a user of this library has it do, as cases to be measured.

A case names a public call and its sizes:

  forward    Kmv.kmv_forward, one product A(theta) V
  step       autograd.kmv and its backward: Y, dL/dtheta and dL/dV (a training step)
  cg         Kmv.kmv_cg_solve, A(theta_s) x = y for every system
  leapfrog   Kmv.leapfrog_step, one step of the HMC map for every system
  phi        Kmv.phi_refresh, the Gibbs draw phi = A^{-1/2} xi by 15 poles
  nystrom    Kmv.nystrom_build, the randomized factorisation of the preconditioner
  update     sampler.hmc_update, one whole update of Algorithm 1, preconditioned
  implicit   Kmv.implicit_step, one preconditioned implicit midpoint step

`inst` instances of `n_lo` to `n` points (log-spaced sizes, so ragged and off
every tile size; one instance has n points), `chains` hyperparameter sets each.
`data` is the distribution of the points, lengthscales and noise:

  line     x ~ U[0,1], y = sin 2 pi x + noise, sigma^2 = 0.01, l ~ 0.2
  normal   x ~ N(0, I_d), l log-uniform in [0.3, 3], sigma^2 = 0.05
  box      x ~ U[-1,1]^d, l log-uniform in [0.5, 5], sigma^2 = 0.05
  unit     x ~ U[0,1]^d, l log-uniform in [0.3, 3], sigma^2 = 0.05, chains jittered
  narrow   x ~ U[0,1]^d, 2 l^2 = (n / 1e4)^(-2/d), sigma^2 = 0.1, chains jittered
  cheb     x ~ U[-1,1]^d, Chebyshev log-amplitude with `cheb` terms per
           dimension, l log-uniform in [0.3, 1], sigma^2 = 0.05
"""
import math

import numpy as np
import torch

from paper_2412_20884_gb300 import Kmv, Points
from paper_2412_20884_gb300.autograd import kmv
from paper_2412_20884_gb300.sampler import hmc_update

N_POLES = 15
CG_TOL = 1e-6


def _case(name, call, n, d, m=1, chains=1, inst=1, n_lo=0, prec="fp32", data="unit", ard=True, cheb=0, rank=0,
          n_int=0, dt=0.0):
    c = dict(call=call, n=n, d=d, m=m, chains=chains, inst=inst, n_lo=n_lo or n, prec=prec, data=data, ard=ard,
             cheb=cheb, rank=rank, n_int=n_int, dt=dt)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one matrix-vector product on a small data set: the smallest call, all latency
        _case("forward_small_fp32", "forward", 2048, 1, data="line", ard=False),
        # the benchmark's training step: product and adjoint over 16 vectors in the tensor-core form
        _case("step_bf16", "step", 65536, 8, m=16, prec="bf16_hilo", data="normal"),
        # the many-dimension, many-vector step, at a size off every tile
        _case("step_wide_bf16", "step", 100000, 32, m=64, prec="bf16_hilo", data="box"),
        # the same kind of step in the default precision
        _case("step_fp32", "step", 20000, 8, m=16, data="normal"),
        # the step of the non-stationary kernel family (64 amplitude coefficients)
        _case("step_cheb_bf16", "step", 65536, 2, m=16, prec="bf16_hilo", data="cheb", ard=False, cheb=8),
        # solves for 8 chains on one mid-sized data set: the tensor-core product with one column
        _case("cg_chains_bf16", "cg", 16384, 3, chains=8, prec="bf16_hilo", data="narrow"),
        # an HMC step on one small data set, in the default precision: launches count
        _case("leapfrog_small_fp32", "leapfrog", 2048, 1, data="line", ard=False, dt=0.01),
        # an HMC step on a batch of independent data sets of mixed sizes, 4 chains each
        _case("leapfrog_batch_bf16", "leapfrog", 16000, 4, chains=4, inst=8, n_lo=1000, prec="bf16_hilo", data="unit",
              dt=0.01),
        # the Gibbs draw without a preconditioner: one multi-shift solve for all poles
        _case("phi_fp32", "phi", 4096, 2, chains=2, data="unit"),
        # the preconditioner's factorisation, rebuilt every few updates
        _case("nystrom_fp32", "nystrom", 16384, 3, chains=8, data="narrow", rank=128),
        # one whole preconditioned update of Algorithm 1 (draw, two energies, 5 leapfrog steps, test)
        _case("update_bf16", "update", 8192, 3, chains=8, prec="bf16_hilo", data="narrow", rank=64, n_int=5, dt=3e-4),
        # the implicit midpoint step: about a hundred products and adjoints on one small data set
        _case("implicit_fp32", "implicit", 2048, 1, data="line", ard=False, rank=64, dt=0.01),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["forward", "forward", "step", "step", "step", "cg", "leapfrog", "leapfrog", "phi", "nystrom",
                       "update", "implicit"])
    prec = rng.choice(["fp32", "bf16_hilo"])
    if call in ("forward", "step"):
        kind = rng.choice(["normal", "box", "unit", "line", "cheb"])
        ard, cheb = rng.random() < 0.7, 0
        d = 1 if kind == "line" else _between(rng, 1, 32)
        m = _between(rng, 1, 64)
        if kind == "cheb":
            d = rng.randint(1, 3)
            cheb = rng.randint(1, (32, 12, 6)[d - 1])
        chains = rng.choice([1, 1, 1, 2, 4])
        inst = rng.choice([1, 1, 1, 2, 5])
        # the multiply-adds of the whole call stay below the largest listed ones of its form
        ops = (d + m) * (1 if call == "forward" else 3 if not cheb else 5) * chains * inst
        most = math.sqrt((3e11 if prec == "fp32" else 2e12) / ops)
        n = _between(rng, 100, max(200.0, min(131072.0, most)))
        return _case("", call, n, d, m=m, chains=chains, inst=inst, n_lo=max(1, n // 8), prec=prec, data=kind,
                     ard=ard, cheb=cheb)
    if call == "nystrom":
        return _case("", call, _between(rng, 1000, 16384), rng.randint(1, 4), chains=rng.randint(1, 8), prec=prec,
                     data=rng.choice(["narrow", "unit"]), rank=rng.randint(16, 128))
    if call == "update":
        return _case("", call, _between(rng, 1000, 8192), rng.randint(2, 4), chains=rng.randint(1, 8), prec=prec,
                     data="narrow", rank=rng.randint(32, 128), n_int=rng.randint(2, 5), dt=rng.uniform(1e-4, 4e-4))
    if call == "implicit":
        return _case("", call, _between(rng, 500, 4096), 1, prec="fp32", data="line", ard=False,
                     rank=rng.randint(48, 96), dt=rng.uniform(0.002, 0.01))
    inst = rng.choice([1, 1, 1, 4, 8]) if call != "phi" else rng.choice([1, 1, 3])
    kind = rng.choice(["unit", "narrow", "line"])
    d = 1 if kind == "line" else rng.randint(2, 4)
    chains = rng.randint(1, 4)
    most = 4096.0 if kind == "line" else 12000.0
    n = _between(rng, 300, min(most, math.sqrt((1.2e9 if prec == "fp32" else 2.4e9) / (chains * inst))))
    return _case("", call, n, d, chains=chains, inst=inst, n_lo=max(100, n // 10), prec=prec, data=kind,
                 ard=kind != "line", dt=rng.uniform(0.002, 0.01))


# ------------------------------------------------------------------------------------------- inputs

def _offsets(case):
    n, lo, k = case["n"], case["n_lo"], case["inst"]
    if k == 1:
        return [0, n]
    sizes = [int(round(lo * (n / lo) ** (b / (k - 1)))) for b in range(k)]
    return [0] + [int(v) for v in np.cumsum(sizes)]


def _inputs(case, seed):
    """Points, observations, hyperparameters and vectors, from the seed alone."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(1000003 * seed + 17)
    h = np.random.default_rng(seed)
    d, chains, kind = case["d"], case["chains"], case["data"]
    off = _offsets(case)
    n, k, cheb = off[-1], case["d"] if case["ard"] else 1, case["cheb"]
    if kind == "normal":
        x = torch.randn(n, d, generator=g, device=dev)
    else:
        x = torch.rand(n, d, generator=g, device=dev)
        if kind in ("box", "cheb"):
            x = 2.0 * x - 1.0
    noise = {"line": 0.1, "narrow": 0.05}.get(kind, 0.1)
    y = torch.sin(2.0 * math.pi * x).sum(dim=1) + noise * torch.randn(n, generator=g, device=dev)
    sigma2 = {"line": 0.01, "narrow": 0.1}.get(kind, 0.05)
    rows = []
    for b in range(case["inst"]):
        nb = off[b + 1] - off[b]
        lo, hi = {"normal": (0.3, 3.0), "box": (0.5, 5.0), "unit": (0.3, 3.0), "cheb": (0.3, 1.0)}.get(kind, (1.0, 1.0))
        base = np.exp(h.uniform(math.log(lo), math.log(hi), k))
        if kind == "line":
            base = np.full(k, 0.2)
        if kind == "narrow":
            base = np.full(k, math.sqrt(0.5 * (nb / 1e4) ** (-2.0 / d)))
        for _ in range(chains):
            if cheb:
                deg = np.indices((cheb,) * d).reshape(d, -1).sum(axis=0)
                head = 0.3 * h.standard_normal(deg.size) / (1.0 + deg)
            else:
                head = np.zeros(1)
            t = np.concatenate([head, np.log(base), [math.log(sigma2)]])
            rows.append(t + (0.0 if cheb else 0.02 * h.standard_normal(t.shape)))
    theta = torch.tensor(np.stack(rows), dtype=torch.float64, device=dev)
    V = torch.randn(chains, n, case["m"], generator=g, device=dev)
    G = torch.randn(chains, n, case["m"], generator=g, device=dev)
    pi = torch.tensor(h.standard_normal(theta.shape), dtype=torch.float64, device=dev)
    return dict(x=x.contiguous(), off=off, y=y, theta=theta, V=V, G=G, pi=pi, gen=g)


def _dense32(x, theta):
    """alpha K0 of one system, FP32, from direct differences."""
    ell = theta[1:-1].exp().float()
    xs = x / ell
    r = torch.cdist(xs, xs, compute_mode="donot_use_mm_for_euclid_dist")
    return theta[0].exp().float() * torch.exp(-0.5 * r * r)


def _phi_draw(case, I):
    """phi ~ N(0, A^{-1}) for every system, as the sampler has it before a step: L^{-T} z with A = L L^T."""
    chains, off = case["chains"], I["off"]
    phi = torch.randn(chains, off[-1], generator=I["gen"], device=I["x"].device)
    for b in range(case["inst"]):
        r = slice(off[b], off[b + 1])
        for c in range(chains):
            th = I["theta"][b * chains + c]
            A = _dense32(I["x"][r], th)
            A = A.double() if A.shape[0] <= 4096 else A   # the large ones in 32 bits, for time
            A.diagonal().add_(th[-1].exp().to(A.dtype))
            L, _ = torch.linalg.cholesky_ex(A)
            z = phi[c, r].to(A.dtype).unsqueeze(1)
            phi[c, r] = torch.linalg.solve_triangular(L.mT, z, upper=True).squeeze(1).float()
    return phi


def _factors(case, I):
    """A rank-r factorisation U diag(lam) U^T of every system's kernel, as the sampler keeps it from an earlier theta."""
    chains, off, rank = case["chains"], I["off"], case["rank"]
    U = torch.zeros(chains, rank, off[-1], device=I["x"].device)
    lam = torch.zeros(case["inst"] * chains, rank, dtype=torch.float64, device=I["x"].device)
    for b in range(case["inst"]):
        r = slice(off[b], off[b + 1])
        for c in range(chains):
            s = b * chains + c
            K = _dense32(I["x"][r], I["theta"][s])
            om = torch.randn(K.shape[0], rank, generator=I["gen"], device=K.device)
            Q, _ = torch.linalg.qr((K @ om).double())
            T = Q.mT @ (K @ Q.float()).double()
            ev, W = torch.linalg.eigh(0.5 * (T + T.mT))
            U[c, :, r] = (Q @ W.flip(1)).float().mT
            lam[s] = ev.flip(0).clamp_min(0.0)
    return U, lam


def prepare(case, seed):
    I = _inputs(case, seed)
    call, chains, n = case["call"], case["chains"], I["off"][-1]
    s = dict(case=case, h=Kmv(0), pts=Points(I["x"], I["off"], ard=case["ard"], cheb=case["cheb"]), theta=I["theta"])
    if call in ("forward", "step"):
        s.update(V=I["V"], G=I["G"])
        if call == "step":
            s["theta"].requires_grad_(True)
            s["V"].requires_grad_(True)
        return s
    s.update(y=I["y"], pi=I["pi"])
    if call in ("leapfrog", "implicit"):
        s["phi"] = _phi_draw(case, I)
    if call in ("phi", "update"):
        s["xi"] = torch.randn(chains, n, generator=I["gen"], device=I["x"].device)
    if call == "nystrom":
        s["omega"] = torch.randn(chains, n, case["rank"], generator=I["gen"], device=I["x"].device)
    elif case["rank"]:
        U, lam = _factors(case, I)
        s["h"].set_preconditioner(s["pts"], U, lam)
    if call == "update":
        s["u"] = 1.0 - torch.rand(s["theta"].shape[0], dtype=torch.float64, generator=I["gen"], device=I["x"].device)
    if call == "implicit":
        s["x0"] = torch.zeros(chains, n, device=I["x"].device)
    return s


# ------------------------------------------------------------------------------------------- the calls

def run(s):
    case, h, pts = s["case"], s["h"], s["pts"]
    call, prec = case["call"], case["prec"]
    if call == "forward":
        return h.kmv_forward(pts, s["theta"], s["V"], prec=prec)
    if call == "step":
        Y = kmv(s["theta"], s["V"], pts, prec, h)
        g_theta, g_V = torch.autograd.grad(Y, (s["theta"], s["V"]), s["G"])
        return Y.detach(), g_theta, g_V
    if call == "cg":
        return h.kmv_cg_solve(pts, s["theta"], s["y"], tol=CG_TOL, maxiter=2000, prec=prec)
    if call == "phi":
        return h.phi_refresh(pts, s["theta"], s["xi"], n_poles=N_POLES, cg_tol=CG_TOL, cg_maxiter=2000, prec=prec)
    if call == "nystrom":
        return h.nystrom_build(pts, s["theta"], s["omega"], prec=prec)
    # the calls that move theta and pi in place start from the state's own
    theta, pi = s["theta"].clone(), s["pi"].clone()
    if call == "leapfrog":
        status, iters, x = h.leapfrog_step(pts, s["y"], s["phi"], theta, pi, case["dt"], cg_tol=CG_TOL,
                                           cg_maxiter=2000, prec=prec)
        return theta, pi, x, status, iters
    if call == "implicit":
        x = s["x0"].clone()
        status, iters, x = h.implicit_step(pts, s["y"], s["phi"], theta, pi, case["dt"], tol=1e-5, maxiter=2000,
                                           x_work=x, prec=prec)
        return theta, pi, x, status, iters
    accepted, fail = hmc_update(h, pts, s["y"], theta, case["dt"], case["n_int"], s["xi"], pi, s["u"], prec=prec,
                                cg_tol=CG_TOL)
    return theta, accepted, fail


def work(case):
    """Bytes: inputs read and outputs written once.  Operations of one pass over the pairs: the distance (2 d), the
    exponential (1) and the multiply-adds of what the call forms from it; the solves count a typical number of
    iterations of their data (what a solve takes depends on its hyperparameters)."""
    off = _offsets(case)
    sizes = np.diff(off).astype(float)
    n, c, d, m = off[-1], case["chains"], case["d"], case["m"]
    pairs = float((sizes * sizes).sum()) * c
    nt = 2 + d
    product = lambda cols: pairs * (2 * d + 1 + 2 * cols)  # noqa: E731
    # the adjoint's sums run over symmetric pairs: half of them
    adjoint = lambda cols: 0.5 * pairs * (2 * d + 1 + 4 * cols + 2 * (2 * d + 1))  # noqa: E731
    vec = 4.0 * n * c
    call = case["call"]
    if call == "forward":
        return {"bytes": 4.0 * n * d + 2 * m * vec, "flops": product(m)}
    if call == "step":
        extra = 2 * product(m) if case["cheb"] else 0.0
        return {"bytes": 4.0 * n * d + 4 * m * vec, "flops": 2 * product(m) + adjoint(m) + extra}
    its = {"line": 45, "unit": 250, "narrow": 210}.get(case["data"], 200)
    if call == "cg":
        return {"bytes": 4.0 * n * (d + 1) + vec, "flops": its * product(1)}
    if call == "leapfrog":
        return {"bytes": 4.0 * n * (d + 1) + 2 * vec + 32.0 * c * nt, "flops": its * product(1) + adjoint(2)}
    if call == "phi":
        return {"bytes": 4.0 * n * d + 2 * vec, "flops": (1 + its) * product(1)}
    r = case["rank"]
    if call == "nystrom":
        return {"bytes": 4.0 * n * d + 2 * r * vec, "flops": product(r) + 4.0 * n * c * 2 * r * r}
    if call == "update":
        pre = 10
        per = pre * (product(1) + 4.0 * n * c * r)
        return {"bytes": 4.0 * n * (d + 1) + (2 + r) * vec,
                "flops": (2 + case["n_int"]) * per + case["n_int"] * adjoint(2) + 2 * product(1) + pre * product(N_POLES)}
    its = 120
    return {"bytes": 4.0 * n * (d + 1) + (3 + r) * vec, "flops": its * (product(1) + adjoint(2) + 4.0 * n * c * r)}


# ------------------------------------------------------------------------------------------- 64-bit values

class _System:
    """One system in 64 bits: rows of K0 scaled by the amplitudes, block by block."""

    def __init__(self, x, theta, ard, cheb):
        self.x, self.cheb, self.ard = x.double(), cheb, ard
        n, d = x.shape
        k = d if ard else 1
        ell = theta[-1 - k:-1].exp()
        self.ell = ell if ard else ell.expand(d)
        self.s2 = theta[-1].exp()
        if cheb:
            T = [torch.ones_like(self.x), self.x]
            for _ in range(2, cheb):
                T.append(2.0 * self.x * T[-1] - T[-2])
            T = torch.stack(T[:cheb])                        # (cheb, n, d)
            self.feat = T[:, :, 0].mT
            for j in range(1, d):
                self.feat = (self.feat[:, :, None] * T[:, :, j].mT[:, None, :]).reshape(n, -1)
            self.amp = torch.exp(self.feat @ theta[:self.feat.shape[1]])
        else:
            self.amp = (0.5 * theta[0]).exp().expand(n)
        self.xs = self.x / self.ell
        self.xs = self.xs - self.xs.mean(dim=0)
        self.nrm = (self.xs * self.xs).sum(dim=1)
        self.rows = max(1, min(n, int(4e8 / n)))

    def blocks(self):
        n = self.x.shape[0]
        for i in range(0, n, self.rows):
            r = slice(i, min(n, i + self.rows))
            e = self.xs[r] @ self.xs.mT
            e.mul_(2.0).sub_(self.nrm[r, None]).sub_(self.nrm[None]).mul_(0.5).clamp_(max=0.0).exp_()
            yield r, e.mul_(self.amp[r, None]).mul_(self.amp[None])

    def dense(self):
        A = torch.cat([k for _, k in self.blocks()])
        A.diagonal().add_(self.s2)
        return A

    def product(self, V):
        return torch.cat([K @ V for _, K in self.blocks()]) + self.s2 * V

    def adjoint(self, V, G):
        """dL/dtheta and A G of L = sum G o (A V)."""
        d = self.x.shape[1]
        q, KV, KG = 0.0, [], []
        dist = torch.zeros(d, dtype=torch.float64, device=V.device)
        xs2 = self.xs * self.xs
        for r, K in self.blocks():
            KG.append(K @ G)
            if self.cheb:
                KV.append(K @ V)
            K.mul_(G[r] @ V.mT)
            qi = K.sum(dim=1)
            q = q + qi.sum()
            dist += (xs2[r] * qi[:, None]).sum(dim=0) + (K @ xs2).sum(dim=0) - 2.0 * (self.xs[r] * (K @ self.xs)).sum(dim=0)
        KG = torch.cat(KG)
        if self.cheb:
            head = self.feat.mT @ ((G * torch.cat(KV)).sum(dim=1) + (V * KG).sum(dim=1))
        else:
            head = q.reshape(1)
        ls = dist if self.ard else dist.sum().reshape(1)
        return torch.cat([head, ls, (self.s2 * (G * V).sum()).reshape(1)]), KG + self.s2 * G


def _cg64(A, b):
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), r @ r
    stop = 1e-28 * float(rr)
    for it in range(20000):
        q = A @ p
        a = rr / (p @ q)
        x += a * p
        r -= a * q
        new = r @ r
        if it % 50 == 49 and float(new) <= stop:
            break
        p = r + (new / rr) * p
        rr = new
    return x


def _inv_sqrt64(A, z, steps=1000):
    """A^{-1/2} z by Lanczos with full reorthogonalisation."""
    n = z.shape[0]
    k = min(n, steps)
    Q = torch.zeros(k, n, dtype=torch.float64, device=z.device)
    al, be = torch.zeros(k, dtype=torch.float64, device=z.device), torch.zeros(k, dtype=torch.float64, device=z.device)
    nz = z.norm()
    Q[0] = z / nz
    used = k
    for j in range(k):
        w = A @ Q[j]
        al[j] = w @ Q[j]
        for _ in range(2):
            w = w - Q[:j + 1].mT @ (Q[:j + 1] @ w)
        be[j] = w.norm()
        if j + 1 == k or float(be[j]) <= 1e-13 * float(al[0].abs()):
            used = j + 1
            break
        Q[j + 1] = w / be[j]
    T = torch.diag(al[:used]) + torch.diag(be[:used - 1], 1) + torch.diag(be[:used - 1], -1)
    ev, W = torch.linalg.eigh(T)
    return nz * (Q[:used].mT @ (W @ (W[0] / ev.sqrt())))


def _force64(sys, x, phi):
    V = torch.stack([x, phi], dim=1)
    G = torch.stack([-0.5 * x, 0.5 * phi], dim=1)
    return sys.adjoint(V, G)[0]


def _too_long(case):
    """Whether the 64-bit value would take over about 20 seconds (at some 0.5 TFLOP/s and 4 TB/s in 64 bits)."""
    sizes = np.diff(_offsets(case)).astype(float)
    c, d, m = case["chains"], case["d"], case["m"]
    pairs = float((sizes * sizes).sum()) * c
    if case["call"] in ("forward", "step"):
        per = 40 + 2 * d + 2 * m + (0 if case["call"] == "forward" else 4 * d + 4 * m + 40)
        return pairs * per / 5e11 > 15 or pairs * 8 * 12 / 4e12 > 15
    if case["call"] == "update":
        return True
    return sizes.max() > 20000 or pairs * 8 * 1000 / 4e12 > 15


def exact(case, seed):
    if _too_long(case):
        return None
    I = _inputs(case, seed)
    call, chains, off = case["call"], case["chains"], I["off"]
    n, dt = off[-1], case["dt"]
    dev = I["x"].device
    systems = [(b, c, slice(off[b], off[b + 1])) for b in range(case["inst"]) for c in range(chains)]

    def system(b, c, r, theta=None):
        return _System(I["x"][r], I["theta"][b * chains + c] if theta is None else theta, case["ard"], case["cheb"])

    if call in ("forward", "step"):
        V, G = I["V"].double(), I["G"].double()
        Y, gV, gt = torch.empty_like(V), torch.empty_like(V), torch.empty_like(I["theta"])
        for b, c, r in systems:
            s = system(b, c, r)
            Y[c, r] = s.product(V[c, r])
            if call == "step":
                gt[b * chains + c], gV[c, r] = s.adjoint(V[c, r], G[c, r])
        return Y if call == "forward" else (Y, gt, gV)
    y = I["y"].double()
    x = torch.empty(chains, n, dtype=torch.float64, device=dev)
    if call == "cg":
        for b, c, r in systems:
            x[c, r] = _cg64(system(b, c, r).dense(), y[r])
        return x, None, None
    if call == "phi":
        xi = torch.randn(chains, n, generator=I["gen"], device=dev).double()
        for b, c, r in systems:
            x[c, r] = _inv_sqrt64(system(b, c, r).dense(), xi[c, r])
        return x, None, None
    if call == "nystrom":
        om = torch.randn(chains, n, case["rank"], generator=I["gen"], device=dev).double()
        lam = torch.zeros(len(systems), case["rank"], dtype=torch.float64, device=dev)
        for b, c, r in systems:
            s = system(b, c, r)
            Y = s.product(om[c, r]) - s.s2 * om[c, r]
            nu = math.sqrt(Y.shape[0]) * 2.0 ** -52 * float(Y.norm() / om[c, r].norm())
            Yn = Y + nu * om[c, r]
            ev, W = torch.linalg.eigh(om[c, r].mT @ Yn)
            B = Yn @ (W / ev.clamp_min(1e-14 * float(ev[-1])).sqrt())
            lam[b * chains + c] = (torch.linalg.svdvals(B) ** 2 - nu).clamp_min(0.0)
        return None, lam, None
    phi = _phi_draw(case, I).double()
    theta, pi = I["theta"].clone(), I["pi"].clone()
    for b, c, r in systems:
        q = b * chains + c
        th0, pi0 = I["theta"][q], I["pi"][q]
        if call == "leapfrog":
            th = th0 + 0.5 * dt * pi0
            s = system(b, c, r, th)
            x[c, r] = _cg64(s.dense(), y[r])
            pi[q] = pi0 - dt * _force64(s, x[c, r], phi[c, r])
            theta[q] = th + 0.5 * dt * pi[q]
            continue
        for _ in range(200):   # implicit midpoint: plain iteration on (theta_1, pi_1) with exact solves
            s = system(b, c, r, 0.5 * (th0 + theta[q]))
            x[c, r] = torch.cholesky_solve(y[r, None], torch.linalg.cholesky(s.dense()))[:, 0]
            new = pi0 - dt * _force64(s, x[c, r], phi[c, r])
            gap = float((new - pi[q]).abs().max())
            pi[q] = new
            theta[q] = th0 + 0.5 * dt * (pi0 + new)
            if gap <= 1e-12 * (1.0 + float(new.abs().max())):
                break
        else:
            return None
    return theta, pi, x, None, None
