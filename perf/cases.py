"""The work that programs have this library do, as cases that can be timed.

A case is one problem shape with the entry point that a program calls on it: the operator and its adjoint,
SGD steps of the three solvers, the full-gradient solver, the differentiable operator and whole epochs of
many problems.  Shapes are those of the library's own workloads and tests, with odd and ragged sizes among
them.  Wavefields are seeded stand-ins with the geometry of a line survey: a direct arrival with free-surface
multiples (down-going), hyperbolic events with noise (up-going), 4 ms sampling, a 20 Hz Ricker wavelet.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2202_04486_gb300 import binding
from paper_2202_04486_gb300.autograd import mdc, reciprocity

DT, F0 = 0.004, 20.0
MU = 0.9


def listed():
    return [
        # a first model on a short line: every launch counts
        dict(name="sgd_nt128_n32", kind="sgd", nt=128, nr=32, nv=32, ns=32, nb=8, steps=4, prec="fp32", recip=False, sym=False, gemv=False),
        # one virtual source on a field-sized line (a target-oriented deconvolution), matrix-vector products
        dict(name="sgd_nt1024_nr180_nv1", kind="sgd", nt=1024, nr=180, nv=1, ns=110, nb=16, steps=4, prec="fp32", recip=False, sym=False, gemv=True),
        # the synthetic ocean-bottom line in plain FP32 with reciprocity, from a symmetric (zero) start
        dict(name="sgd_nt512_n201_sym", kind="sgd", nt=512, nr=201, nv=201, ns=201, nb=16, steps=4, prec="fp32", recip=True, sym=True, gemv=False),
        # modelling with a given reflection response: the operator alone, split-BF16 products
        dict(name="forward_nt1024_n301", kind="forward", nt=1024, nr=301, nv=301, ns=401, nb=32, prec="bf16x3"),
        # imaging by cross-correlation, or a solver of the user's own: the adjoint alone
        dict(name="adjoint_nt1024_n301", kind="adjoint", nt=1024, nr=301, nv=301, ns=401, nb=32, prec="bf16x3"),
        # stochastic steps of the mixed-precision workload
        dict(name="sgd_nt1024_n301", kind="sgd", nt=1024, nr=301, nv=301, ns=401, nb=32, steps=3, prec="bf16x3", recip=False, sym=False, gemv=False),
        # the same problem in plain FP32, the larger batch
        dict(name="sgd_nt1024_n301_nb64_fp32", kind="sgd", nt=1024, nr=301, nv=301, ns=401, nb=64, steps=2, prec="fp32", recip=False, sym=False, gemv=False),
        # the differentiable operator under a preconditioner written in torch: prediction and model gradient
        dict(name="autograd_nt512_n256", kind="autograd", nt=512, nr=256, nv=256, ns=256, nb=16, prec="fp32"),
        # momentum and causality mute on odd sizes (unaligned traces, ragged tiles, an odd batch)
        dict(name="nsgd_nt750_ragged", kind="nsgd", nt=750, nr=237, nv=133, ns=190, nb=27, steps=3, prec="fp32", recip=False),
        # the full-gradient solver that the stochastic one is compared with: every source in one batch
        dict(name="lsqr_nt512_n201", kind="lsqr", nt=512, nr=201, nv=201, ns=201, iters=2, prec="fp32", recip=True),
        # a long record on a large square array with reciprocity (FFT length 3072), symmetric start
        dict(name="sgd_nt1500_n600_sym", kind="sgd", nt=1500, nr=600, nv=600, ns=300, nb=32, steps=2, prec="bf16x3", recip=True, sym=True, gemv=False),
        # one epoch of seven surveys of uneven sizes, replayed from the captured graph
        dict(name="epoch_7_surveys", kind="epoch", members=7, base=1000, nb=32, branches=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sgd", "sgd", "sgd", "nsgd", "forward", "adjoint", "autograd", "lsqr", "epoch"])
    if kind == "epoch":
        while True:
            case = dict(kind="epoch", members=rng.randint(2, 5), base=rng.randint(2000, 900000), nb=rng.choice([16, 32, 32, 48]), branches=rng.choice([2, 4, 8]))
            if work(case)["bytes"] <= 0.6 * work(listed()[-1])["bytes"]:
                return case
    prec = rng.choice(["fp32", "bf16x3"])
    while True:
        nt = rng.choice([128, 256, 512, 1024, 1500]) if rng.random() < 0.5 else _log_int(rng, 100, 1500)
        nr, nv, ns = _log_int(rng, 24, 600), _log_int(rng, 24, 600), _log_int(rng, 24, 500)
        if kind == "autograd" or rng.random() < 0.3:
            nv = nr
        nb = min(ns, _log_int(rng, 4, 64))
        if nr * nv * nt <= 2.0e8 and ns * nr * nt <= 2.0e8 and ns * nv * nt <= 2.0e8 and (kind != "lsqr" or ns * nr * nv * nt <= 8.0e9):
            break
    case = dict(kind=kind, nt=nt, nr=nr, nv=nv, ns=ns, prec=prec)
    if kind == "lsqr":
        return dict(case, iters=rng.randint(1, 3), recip=nr == nv)
    case["nb"] = nb
    if kind in ("sgd", "nsgd"):
        case.update(steps=rng.randint(1, 4), recip=nr == nv)
    if kind == "sgd":
        case.update(sym=nr == nv and rng.random() < 0.5, gemv=False)
    return case


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _members(case):
    """Uneven survey shapes as the many-problem workload draws them (reciprocity where the array is square)."""
    out = []
    for i in range(case["members"]):
        r = np.random.default_rng(case["base"] + i)
        nt = int(r.choice([256, 512, 1024, 1500]))
        nr, nv, ns = int(r.integers(64, 601)), int(r.integers(64, 601)), int(r.integers(64, 801))
        out.append(dict(kind="sgd", nt=nt, nr=nr, nv=nv, ns=ns, nb=min(case["nb"], ns), steps=-(-ns // case["nb"]), prec="bf16x3",
                        recip=nr == nv, sym=False, gemv=False))
    return out


def _events(n1, n2, nt, g, t0, amp, vel, gain, noise):
    """Sum of hyperbolic Ricker events [n1][n2][nt] float32 with a gain per first index and white noise."""
    dev = "cuda"
    t = torch.arange(nt, device=dev, dtype=torch.float32) * DT
    out = torch.empty((n1, n2, nt), device=dev)
    rows = max(1, (1 << 26) // (n2 * nt))
    for a in range(0, n1, rows):
        b = min(n1, a + rows)
        h = 20.0 * (torch.arange(n2, device=dev)[None, :] - torch.arange(a, b, device=dev)[:, None]).float()
        acc = out[a:b]
        acc.normal_(generator=g).mul_(noise)
        for k in range(len(t0)):
            arrival = torch.sqrt(t0[k] ** 2 + (h / vel[k]) ** 2)
            x = (math.pi * F0 * (t[None, None, :] - arrival[:, :, None])).square_()
            acc.add_((1.0 - 2.0 * x).mul_(torch.exp(-x)), alpha=float(amp[k]))
        acc.mul_(gain[a:b, None, None])
    return out


def _step_size(D):
    """1 / sigma^2 of the kernel, from a few bins of the wavelet's band."""
    ns, nr, nt = D.shape
    ph = 2 * math.pi * DT * torch.arange(nt, device="cuda", dtype=torch.float64)[:, None] * torch.arange(5, 45, 3, device="cuda", dtype=torch.float64)[None, :]
    K = torch.complex(D.reshape(-1, nt) @ ph.cos().float(), D.reshape(-1, nt) @ ph.sin().float())
    K = K.reshape(ns, nr, -1).permute(2, 0, 1).contiguous()
    x = torch.ones((K.shape[0], nr, 1), device="cuda", dtype=K.dtype)
    for _ in range(12):
        y = K.mH @ (K @ x)
        lam = torch.linalg.vector_norm(y, dim=(1, 2), keepdim=True)
        x = y / lam
    return 0.7 / float(lam.max())


def _inputs(case, seed):
    """What the program has in hand, from the seed alone: kernel D, data or model, batches, step size."""
    nt, nr, nv, ns = case["nt"], case["nr"], case["nv"], case["ns"]
    rng = np.random.default_rng(seed)
    g = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 40)))
    td, delta = rng.uniform(0.05, 0.07), rng.uniform(0.18, 0.22) * nt * DT
    gain = lambda n: torch.from_numpy(rng.uniform(0.8, 1.2, n).astype(np.float32)).cuda()
    orders = range(5)
    D = _events(ns, nr, nt, g, [td + m * delta for m in orders], [(-0.5) ** m for m in orders], [1500.0] * 5, gain(ns), 0.005)
    hyper = lambda: (rng.uniform(0.15, 0.85, 8) * nt * DT, rng.uniform(0.2, 1.0, 8), rng.uniform(1500.0, 2500.0, 8))
    d = dict(D=D)
    nb = case.get("nb", ns)
    perm = rng.permutation(ns).astype(np.int32)
    steps = case.get("steps", 1)
    d["perm"] = perm
    order = np.resize(perm, max(ns, steps * nb))
    last = steps * nb > ns and -(-ns // nb) == steps   # a whole epoch ends with a partial batch
    d["batches"] = [(perm if last else order)[k * nb:(k + 1) * nb] for k in range(steps)]
    if case["kind"] in ("forward", "autograd"):
        X = _events(nv, nr, nt, g, *hyper(), gain(nv), 0.01)
        d["X"] = X
    if case["kind"] == "adjoint":
        d["R"] = _events(nb, nv, nt, g, *hyper(), gain(nb), 0.05)
    elif case["kind"] == "autograd":
        d["W"] = _events(nb, nv, nt, g, *hyper(), gain(nb), 0.05)
    elif case["kind"] != "forward":
        d["U"] = _events(ns, nv, nt, g, *hyper(), gain(ns), 0.05)
        d["alpha"] = _step_size(D)
    if case["kind"] == "nsgd":
        h = 20.0 * np.abs(np.arange(nr)[None, :] - np.arange(nv)[:, None])
        d["mute"] = np.clip(np.floor((h / 2500.0 - 1.5 / F0) / DT), 0, nt).astype(np.int32)
    return d


def _plan(case, D, nb_max):
    plan = binding.MDCPlan(D, case["nv"], nb_max=nb_max,
                           precision=binding.MDC_PREC_BF16X3 if case["prec"] == "bf16x3" else binding.MDC_PREC_FP32)
    if case.get("gemv"):
        plan.set_config(gemm_fwd=binding.MDC_GEMM_GEMV, gemm_adj=binding.MDC_GEMM_GEMV)
    return plan


def prepare(case, seed):
    kind = case["kind"]
    if kind == "epoch":
        members, keep = [], []
        for i, m in enumerate(_members(case)):
            d = _inputs(m, seed + 7919 * i)
            members.append(dict(plan=_plan(m, d["D"], m["nb"]), X=torch.zeros((m["nv"], m["nr"], m["nt"]), device="cuda"), U_obs=d["U"],
                                perm=torch.from_numpy(d["perm"][None, :]).cuda(), nb=m["nb"], alpha=d["alpha"],
                                flags=binding.SMDD_RECIPROCITY if m["recip"] else 0,
                                loss=torch.zeros((1, m["steps"]), device="cuda", dtype=torch.float64)))
        torch.cuda.synchronize()
        return dict(kind=kind, batch=binding.MDCBatch(members, n_branches=case["branches"]), members=members)
    d = _inputs(case, seed)
    nt, nr, nv, ns = case["nt"], case["nr"], case["nv"], case["ns"]
    st = dict(kind=kind, case=case, plan=_plan(case, d["D"], case.get("nb", ns)),
              idx=[torch.from_numpy(b).cuda() for b in d["batches"]])
    if kind in ("forward", "autograd"):
        st["X"] = d["X"]
    if kind == "adjoint":
        st["R"] = d["R"]
    if kind == "autograd":
        st["W"] = d["W"]
    if kind in ("sgd", "nsgd", "lsqr"):
        st.update(X=torch.zeros((nv, nr, nt), device="cuda"), U=d["U"], alpha=d["alpha"])
        st["flags"] = binding.SMDD_RECIPROCITY if case["recip"] else 0
    if kind in ("sgd", "nsgd"):
        st["flags"] |= binding.SMDD_KEEP_XHAT | binding.SMDD_REUSE_XHAT | (binding.SMDD_SYMMETRIC if case.get("sym") else 0)
        st["loss"] = torch.zeros(case["steps"], device="cuda", dtype=torch.float64)
        st["losses"] = list(st["loss"].split(1))
    if kind == "nsgd":
        st.update(V=torch.zeros_like(st["X"]), mute=torch.from_numpy(d["mute"]).cuda())
    if kind == "lsqr":
        st["norms"] = torch.zeros(case["iters"] + 1, device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    return st


def run(st):
    kind = st["kind"]
    if kind == "epoch":
        st["batch"].run(0, 1)
        return [[m["X"], m["loss"].float()] for m in st["members"]]   # losses are logged in single precision
    plan = st["plan"]
    if kind == "sgd":
        for idx, loss in zip(st["idx"], st["losses"]):
            plan.step(st["X"], st["U"], idx, st["alpha"], st["flags"], loss)
        return st["X"], st["loss"].float()
    if kind == "nsgd":
        for idx, loss in zip(st["idx"], st["losses"]):
            plan.step_nsgd(st["X"], st["V"], st["U"], idx, st["alpha"], MU, st["flags"], st["mute"], loss)
        return st["X"], st["V"], st["loss"].float()
    if kind == "forward":
        return plan.forward(st["X"], st["idx"][0])
    if kind == "adjoint":
        return plan.adjoint(st["R"], st["idx"][0])
    if kind == "lsqr":
        st["X"].zero_()
        plan.lsqr(st["X"], st["U"], st["case"]["iters"], st["flags"], norms=st["norms"])
        return st["X"], st["norms"].float()
    X = st["X"].detach().requires_grad_(True)
    U = mdc(reciprocity(X), plan, st["idx"][0])
    (G,) = torch.autograd.grad(U, X, st["W"])
    return U.detach(), G


# ------------------------------------------------------------------------------------------------
# work and exact values
# ------------------------------------------------------------------------------------------------
def work(case):
    """Products of 8 flops a complex multiply-add over the bins of an FFT of 2 nt samples, 2.5 N log2 N flops a
    real transform; the model, the batch rows of the kernel spectra and of the data once each."""
    kind = case["kind"]
    if kind == "epoch":
        w = [work(m) for m in _members(case)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    nt, nr, nv, ns = case["nt"], case["nr"], case["nv"], case["ns"]
    nb, N, nf = case.get("nb", ns), 2 * nt, nt + 1
    fft, one, model, rows, data = 2.5 * N * math.log2(N), 8.0 * nf * nb * nr * nv, 4.0 * nv * nr * nt, 8.0 * nf * nb * nr, 4.0 * nb * nv * nt
    if kind in ("forward", "adjoint"):
        return {"bytes": model + rows + data, "flops": one + fft * (nr * nv + nb * nv)}
    if kind == "autograd":
        return {"bytes": 2 * model + rows + 2 * data, "flops": 2 * one + 2 * fft * (nr * nv + nb * nv)}
    if kind == "lsqr":
        n = case["iters"]
        return {"bytes": model + rows + data + n * (6 * model + 2 * rows + 2 * data),
                "flops": (2 * n + 1) * (one + fft * (nr * nv + nb * nv))}
    traces = nv * (nv + 1) / 2 if case.get("sym") else nr * nv
    state = 1.0 if kind == "sgd" else 2.0
    total = {"bytes": 0.0, "flops": 0.0}
    left = ns if case["steps"] * nb > ns and -(-ns // nb) == case["steps"] else case["steps"] * nb
    for _ in range(case["steps"]):
        b = min(nb, left) / nb
        left -= nb
        total["bytes"] += state * model * (1.0 + traces / (nr * nv)) + b * (rows + data)
        total["flops"] += 2 * b * one + 2 * fft * (traces + b * nb * nv)
    return total


class _Exact:
    """The operator in 64 bits: FFT of 2 nt samples, one product per frequency, causal window."""

    def __init__(self, D):
        self.nt = D.shape[2]
        self.n = 2 * self.nt
        self.K = self.spectra(D)

    def spectra(self, x):
        return torch.fft.rfft(x.double(), n=self.n).permute(2, 0, 1).contiguous()

    def window(self, S):
        return torch.fft.irfft(S.permute(1, 2, 0).contiguous(), n=self.n)[:, :, :self.nt].contiguous()

    def forward(self, X, idx):
        X = self.spectra(X)
        return self.window(self.K[:, idx] @ X.mT)

    def adjoint(self, R, idx):
        R = self.spectra(R)
        return self.window(R.mT @ self.K[:, idx].conj())


def _sym(G):
    return 0.5 * (G + G.transpose(0, 1))


def _exact_steps(case, d):
    A = _Exact(d["D"])
    X = torch.zeros((case["nv"], case["nr"], case["nt"]), device="cuda", dtype=torch.float64)
    V, losses, alpha = torch.zeros_like(X), [], float(np.float32(d["alpha"]))
    keep = None
    if case["kind"] == "nsgd":
        keep = torch.arange(case["nt"], device="cuda")[None, None, :] >= torch.from_numpy(d["mute"]).cuda()[:, :, None]
    mu = float(np.float32(MU))
    for b in d["batches"]:
        idx = torch.from_numpy(b).cuda().long()
        R = A.forward(X, idx) - d["U"][idx].double()
        losses.append(0.5 * (R * R).sum())
        G = A.adjoint(R, idx)
        if case["recip"]:
            G = _sym(G)
        if case["kind"] == "nsgd":
            G = G * keep
            V = mu * V - alpha * G
            X = X + mu * V - alpha * G
        else:
            X = X - alpha * G
    return X, V, torch.stack(losses)


def _exact_lsqr(case, d):
    """LSQR (Paige & Saunders 1982) from zero on the operator with the reciprocity projection."""
    A = _Exact(d["D"])
    idx = torch.arange(case["ns"], device="cuda")
    C = _sym if case["recip"] else (lambda G: G)
    x = torch.zeros((case["nv"], case["nr"], case["nt"]), device="cuda", dtype=torch.float64)
    u = d["U"].double()
    beta = u.norm()
    u = u / beta
    v = C(A.adjoint(u, idx))
    alpha = v.norm()
    v = v / alpha
    w, phibar, rhobar, norms = v, beta, alpha, [beta]
    for _ in range(case["iters"]):
        u = A.forward(v, idx) - alpha * u
        beta = u.norm()
        u = u / beta
        v = C(A.adjoint(u, idx)) - beta * v
        alpha = v.norm()
        v = v / alpha
        rho = torch.hypot(rhobar, beta)
        c, s = rhobar / rho, beta / rho
        theta, rhobar, phi, phibar = s * alpha, -c * alpha, c * phibar, s * phibar
        x = x + (phi / rho) * w
        w = v - (theta / rho) * w
        norms.append(phibar)
    return x, torch.stack(norms)


def exact(case, seed):
    kind = case["kind"]
    if kind == "epoch":
        out = []
        for i, m in enumerate(_members(case)):
            X, _, losses = _exact_steps(m, _inputs(m, seed + 7919 * i))
            out.append([X, losses[None, :]])
        return out
    d = _inputs(case, seed)
    if kind == "lsqr":
        return _exact_lsqr(case, d)
    if kind in ("sgd", "nsgd"):
        X, V, losses = _exact_steps(case, d)
        return (X, losses) if kind == "sgd" else (X, V, losses)
    A, idx = _Exact(d["D"]), torch.from_numpy(d["batches"][0]).cuda().long()
    if kind == "forward":
        return A.forward(d["X"], idx)
    if kind == "adjoint":
        return A.adjoint(d["R"], idx)
    return A.forward(_sym(d["X"].double()), idx), _sym(A.adjoint(d["W"], idx))
