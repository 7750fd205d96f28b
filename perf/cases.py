"""The performance cases: the work a program of this library has it do, through its Python
binding, on inputs made from a seed alone.

A case is a dict of plain values; ``prepare`` makes what a program holds before the call (a
filter with its initial particles and the observations it will be fed, a proposal network
with its rows, resampling weights), ``run`` is one pass and returns what the call gives its
caller, ``work`` counts the bytes and operations no implementation can avoid, and ``exact``
gives the first pass's outputs in 64 bits from the method's definition (Philox4x32-10 words,
Box-Muller normals, the filter's equations in torch), without the library.

A filter pass is one step with one observation: that is how a filter is used, on line. The
step's outputs are the filtered mean and the evidence; the particles stay inside the filter's
handle and are the next pass's input, so a later pass's outputs depend on all of them. The steps of an FP32 filter give their
estimates in single precision here, as a program logs the track of a single-precision
filter (the binding's device outputs are doubles whatever the filter's precision).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1203_2394_gb300 import dpf, workloads

# Observations of a filter: the time terms of the growth map (cos 1.2 t) and of the paper's
# models (sin t as well) come back to their phase after these many steps, so that a program
# that runs longer sees one jump of the state and no lasting mismatch of its model.
T_GROWTH, T_PAPER, T_LINEAR = 1775, 3550, 512


def listed():
    return [
        # a small tracking filter in double precision, one host observation in and one host
        # estimate out: the smallest call, where latency and launches count
        {"name": "online_lg4_f64", "kind": "online", "N": 256, "M": 32, "L": 8},
        # the headline workload: conditionally linear-Gaussian growth model, one step
        {"name": "growth_clg10", "kind": "ladpf", "model": "growth_clg10", "N": 65536, "M": 128, "L": 16},
        # the same model at sizes that are no multiple of anything (the ragged rows' path)
        {"name": "growth_clg10_ragged", "kind": "ladpf", "model": "growth_clg10", "N": 3001, "M": 100, "L": 7},
        # the high-dimensional workload: 56 inner dimensions, dense transition, the largest step
        {"name": "growth_clg64", "kind": "ladpf", "model": "growth_clg64", "N": 32768, "M": 256, "L": 16},
        # the paper's own nonlinear benchmark model 1 (Table 1)
        {"name": "paper_model1", "kind": "paper", "model": 1, "N": 65536, "M": 128, "L": 16},
        # many independent filters of one dimension stepped together, each its own model and sizes
        {"name": "batch_lg16", "kind": "batch", "F": 16, "Nmax": 16384, "mix": 5, "L": 8},
        # the bootstrap particle filter the paper compares with, at the headline's N (M + 1) particles
        {"name": "particle_filter", "kind": "pf", "model": "growth_clg10", "N": 8454144},
        # the decentralized filter without look-ahead, at the headline's sizes
        {"name": "standard_dpf", "kind": "std", "model": "growth_clg10", "N": 65536, "M": 128},
        # the filter with the outer-amortised learned proposal
        {"name": "learned_lg4", "kind": "learned", "N": 262144, "M": 64, "L": 8},
        # the mixture proposal's network over many feature rows (an odd count)
        {"name": "proposal_forward", "kind": "forward", "n": 1000003},
        # one training minibatch of the mixture proposal: loss and gradients, BF16 operands
        {"name": "proposal_gradient", "kind": "grad", "form": "mixture", "bf16": True, "n": 1024},
        # systematic resampling of a weight vector held on the device (an odd count)
        {"name": "resample_global", "kind": "resample", "n": 1000003, "dtype": "f32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["online", "ladpf", "ladpf", "ladpf", "paper", "batch", "pf", "std", "learned",
                       "forward", "grad", "resample"])
    if kind == "online":
        return {"kind": kind, "N": _log_int(rng, 64, 16384), "M": rng.randint(8, 64), "L": rng.randint(2, 16)}
    if kind == "ladpf":
        if rng.random() < 0.35:
            return {"kind": kind, "model": "growth_clg64", "N": _log_int(rng, 512, 32768),
                    "M": rng.choice([64, 100, 128, 192, 256, 256]), "L": rng.choice([4, 8, 16])}
        return {"kind": kind, "model": "growth_clg10", "N": _log_int(rng, 1000, 65536),
                "M": rng.choice([32, 45, 64, 100, 128, 128, 192, 256]), "L": rng.choice([4, 7, 8, 16, 16, 32])}
    if kind == "paper":
        return {"kind": kind, "model": rng.choice([1, 2]), "N": _log_int(rng, 1000, 65536),
                "M": rng.choice([20, 32, 45, 64, 128]), "L": rng.choice([7, 8, 16, 32])}
    if kind == "batch":
        return {"kind": kind, "F": rng.randint(2, 24), "Nmax": _log_int(rng, 1024, 16384),
                "mix": rng.randint(0, 999), "L": rng.choice([4, 8, 16])}
    if kind == "pf":
        return {"kind": kind, "model": rng.choice(["growth_clg10", "lg4"]), "N": _log_int(rng, 10000, 8454144)}
    if kind == "std":
        return {"kind": kind, "model": rng.choice(["growth_clg10", "lg4"]), "N": _log_int(rng, 1000, 65536),
                "M": rng.choice([19, 32, 64, 100, 128, 256])}
    if kind == "learned":
        return {"kind": kind, "N": _log_int(rng, 4096, 262144), "M": rng.choice([32, 64, 128]),
                "L": rng.choice([4, 8, 16])}
    if kind == "forward":
        return {"kind": kind, "n": _log_int(rng, 1000, 1000003)}
    if kind == "grad":
        return {"kind": kind, "form": rng.choice(["mixture", "mixture", "wide"]), "bf16": rng.random() < 0.7,
                "n": _log_int(rng, 256, 16384)}
    return {"kind": kind, "n": _log_int(rng, 1000, 16777216), "dtype": rng.choice(["f32", "f32", "f64"])}


# ---- inputs ----
def _spec(case, seed):
    """The conditionally linear-Gaussian model of a filter case."""
    name = case.get("model") or "lg4"
    return workloads.make_model(name, seed % 1000)


def _observations(spec, seed, dtype):
    T = T_LINEAR if spec.growth is None else T_GROWTH
    return workloads.simulate(spec, T, seed)[1].astype(dtype)


def _batch_members(case, seed):
    """Sizes (by the case alone), models and seeds of a batch's filters."""
    r = np.random.default_rng(case["mix"])
    F = case["F"]
    d1s = [int(v) for v in r.choice([1, 2, 4, 8], F)]
    Ns = [int(v) for v in r.integers(min(1024, case["Nmax"]), case["Nmax"] + 1, F)]
    Ms = [int(v) for v in r.choice([16, 32, 64, 128, 256], F)]
    specs = [workloads.make_model("lg16", 1000 * (seed % 1000) + f, d1s[f]) for f in range(F)]
    return d1s, Ns, Ms, specs, [seed + 7919 * f for f in range(F)]


def _proposal_shape(form):
    """(d1, d2, dy, inputs, head outputs) of a proposal form."""
    if form == "wide":
        return 8, 56, 8, 2 * 8 + 8 + 2 * 56, 2 * 56
    return 2, 2, 2, 8, 20


def _proposal_weights(form, seed):
    """A mixture head near the prior, or an amortised map near the identity (64-bit values that
    are exact in 32 bits, as the library holds them)."""
    d1, d2, dy, din, dout = _proposal_shape(form)
    W = workloads.init_mlp_weights(din, 256, dout, seed=seed % 100000)
    if form == "mixture":
        W["b4"][12:] = np.log(np.sqrt(0.1))
    return {k: v.astype(np.float32).astype(np.float64) for k, v in W.items()}


def _proposal_rows(case, seed):
    """Feature rows, targets and weights of a proposal case, by their law in a filter: states
    and observations of order one, targets near the prior mean, positive skewed weights."""
    form = case.get("form", "mixture")
    d1, d2, dy, din, dout = _proposal_shape(form)
    g = torch.Generator().manual_seed(seed)
    n = case["n"]
    F = torch.randn((n, din), generator=g)
    if form == "wide":
        F[:, din - d2:] = F[:, din - d2:].square() * 0.1  # variances of the group's prior means
        mean = F[:, 2 * d1 + dy:2 * d1 + dy + d2]
        mu = mean + 0.3 * torch.randn((n, d2), generator=g)
        Z = torch.cat([mu + 0.3162 * torch.randn((n, d2), generator=g), mu, mean], 1)
    else:
        Z = 0.8 * F[:, 2 * d1:2 * d1 + d2] + 0.3162 * torch.randn((n, d2), generator=g)
    w = torch.exp(0.7 * torch.randn((n,), generator=g)) / n
    return F, Z, w


def _resample_weights(case, seed):
    """Importance weights of a particle set: log-normal, some of them negligible."""
    g = torch.Generator().manual_seed(seed)
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    w = torch.exp(1.5 * torch.randn((case["n"],), generator=g, dtype=dt))
    u = torch.randint(0, 2 ** 31 - 1, (1,), generator=g, dtype=torch.int32)
    return w, u


def _amortised(seed, lg4):
    p = dpf.Proposal(2, 2, 2, hidden=256, amortised_Qz=lg4.Q[2:, 2:])
    W = workloads.init_mlp_weights(10, 256, 4, seed=seed % 100000)
    W["W4"] *= 0.5  # near the identity map: scales and shifts of a tenth or so
    p.set_weights(W)
    return p


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "k": 0}
    if kind == "online":
        spec = _spec(case, seed)
        st["f"] = dpf.Filter(dpf.Model.from_spec(spec, dpf.DPF_F64), spec.d1, spec.d2, case["N"], case["M"],
                             case["L"], seed)
        st["ys"] = _observations(spec, seed, np.float64)
        return st
    if kind in ("ladpf", "pf", "std", "learned"):
        spec = _spec(case, seed)
        model = dpf.Model.from_spec(spec, dpf.DPF_F32)
        if kind == "pf":
            st["f"] = dpf.ParticleFilter(model, spec.d1, spec.d2, case["N"], seed)
        elif kind == "std":
            st["f"] = dpf.StandardDPF(model, spec.d1, spec.d2, case["N"], case["M"], seed)
        else:
            st["f"] = dpf.Filter(model, spec.d1, spec.d2, case["N"], case["M"], case["L"], seed)
        if kind == "learned":
            st["p"] = _amortised(seed, spec)
            st["f"].set_proposal(st["p"])
        ys = _observations(spec, seed, np.float32)
    elif kind == "paper":
        model = dpf.PaperModel(case["model"])
        st["f"] = dpf.Filter(model, model.d1, model.d2, case["N"], case["M"], case["L"], seed)
        ys = workloads.simulate_paper(case["model"], T_PAPER, seed)[1].astype(np.float32)
    elif kind == "batch":
        d1s, Ns, Ms, specs, seeds = _batch_members(case, seed)
        st["f"] = dpf.Batch([dpf.Model.from_spec(s, dpf.DPF_F32) for s in specs], d1s, Ns, Ms, case["L"], seeds)
        ys = np.stack([workloads.simulate(s, 128, seed + f)[1] for f, s in enumerate(specs)], 1).astype(np.float32)
    elif kind in ("forward", "grad"):
        form = case.get("form", "mixture")
        d1, d2, dy, din, dout = _proposal_shape(form)
        if form == "wide":
            st["p"] = dpf.Proposal(d1, d2, dy, hidden=256, amortised_Qz=0.1 * np.eye(d2))
        else:
            st["p"] = dpf.Proposal(d1, d2, dy, hidden=256, components=4)
        st["p"].set_weights(_proposal_weights(form, seed))
        if kind == "grad" and not case["bf16"]:
            st["p"].set_bf16(False)
        st["rows"] = [t.cuda() for t in _proposal_rows(case, seed)]
        return st
    else:
        w, u = _resample_weights(case, seed)
        st["w"], st["u"] = w.cuda(), u.cuda()
        return st
    st["ys"] = torch.from_numpy(ys).cuda()
    # the estimates' device buffer: the means, then the log-evidence, of one filter or of each
    F = case["F"] if kind == "batch" else 1
    st["nmean"] = F * st["f"].d
    st["out"] = torch.empty(st["nmean"] + F, dtype=torch.float64, device="cuda")
    return st


def run(state):
    kind = state["case"]["kind"]
    if kind == "online":
        y = state["ys"][state["k"] % len(state["ys"])]
        state["k"] += 1
        mean, logz = state["f"].step(y)
        return {"mean": mean, "logz": logz}
    if kind == "forward":
        return {"head": state["p"].forward(state["rows"][0])}
    if kind == "grad":
        loss, g = state["p"].loss_grad(*state["rows"])
        return {"loss": np.float32(loss), "grad": g}
    if kind == "resample":
        return {"index": dpf.resample(state["w"], state["u"])}
    ys, out, nm = state["ys"], state["out"], state["nmean"]
    y = ys[state["k"] % ys.shape[0]]
    state["k"] += 1
    state["f"].step_device(y.data_ptr(), out.data_ptr(), out.data_ptr() + 8 * nm)
    est = out.float()
    return {"mean": est[:nm], "logz": est[nm:]}


# ---- what a pass cannot do without ----
def _step_work(N, M, L, d1, d2, dy, s):
    """One look-ahead step: the inner set and its log-weights read once and written once, the
    outer particle's row, weight, ancestor and choice; the operations of the propagation, the
    y update and the look-ahead's projection (matrix products) and of its L M pairs."""
    by = s * 2 * N * M * (d2 + 1) + N * (2 * d1 * s + 12)
    fl = N * M * (2.0 * d2 * (d2 + d1) + 2 * dy * d2 + 2 * dy * (d1 + d2)) + N * M * L * (3.0 * dy + 3)
    return by, fl


def work(case):
    kind = case["kind"]
    if kind in ("online", "learned"):
        s = 8 if kind == "online" else 4
        by, fl = _step_work(case["N"], case["M"], case["L"], 2, 2, 2, s)
        if kind == "learned":
            fl += 2.0 * case["N"] * (10 * 256 + 2 * 256 * 256 + 256 * 4)
    elif kind == "ladpf":
        d1, d2, dy = (2, 8, 2) if case["model"] == "growth_clg10" else (8, 56, 8)
        by, fl = _step_work(case["N"], case["M"], case["L"], d1, d2, dy, 4)
    elif kind == "paper":
        d = case["model"]
        by, fl = _step_work(case["N"], case["M"], case["L"], d, d, 1, 4)
        fl += case["N"] * case["M"] * (20.0 * d + 4.0 * d * case["L"])
    elif kind == "batch":
        d1s, Ns, Ms, _, _ = _batch_members({**case}, 0)
        parts = [_step_work(N, M, case["L"], d1, 16 - d1, 4, 4) for d1, N, M in zip(d1s, Ns, Ms)]
        by, fl = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "pf":
        d, dy, d2 = (10, 2, 8) if case["model"] == "growth_clg10" else (4, 2, 2)
        by, fl = case["N"] * (2 * 4 * d + 8), case["N"] * (2.0 * d2 * d2 + 2 * dy * d2 + 20)
    elif kind == "std":
        d1, d2, dy = (2, 8, 2) if case["model"] == "growth_clg10" else (2, 2, 2)
        by, fl = _step_work(case["N"], case["M"], 0, d1, d2, dy, 4)
    elif kind in ("forward", "grad"):
        d1, d2, dy, din, dout = _proposal_shape(case.get("form", "mixture"))
        params = 256 * (din + 512 + dout) + 768 + dout
        macs = 256 * (din + 512 + dout)
        if kind == "forward":
            by, fl = case["n"] * 4 * (din + dout) + 4 * params, 2.0 * case["n"] * macs
        else:
            zw = 3 * d2 if case["form"] == "wide" else d2
            by, fl = case["n"] * 4 * (din + zw + 1) + 8 * params, 6.0 * case["n"] * macs
    else:
        s = 8 if case["dtype"] == "f64" else 4
        by, fl = case["n"] * (s + 4), 2.0 * case["n"]
    return {"bytes": float(by), "flops": float(fl)}


# ---- the first pass in 64 bits ----
INIT_X, INIT_Z, LA_J, LA_X, LA_Z, PROP, PF_X, PF_Z = 1, 2, 3, 4, 5, 9, 12, 13


def _philox(seed, t, i, purpose, sub, block):
    """Philox4x32-10 (Salmon et al., SC'11) over broadcast counters; four int64 tensors."""
    m32 = 0xFFFFFFFF
    i, sub, block = torch.broadcast_tensors(i, sub, block)
    c = [torch.full_like(i, t), i, sub | (purpose << 24), block]
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # modulo 2^64: the bits are all there
        c = [((p1 >> 32) & m32) ^ c[1] ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _pair(wa, wb):
    r = torch.sqrt(-2.0 * torch.log(((wa >> 9).double() + 0.5) * 2.0 ** -23))
    th = 2.0 * math.pi * ((wb >> 9).double() + 0.5) * 2.0 ** -23
    return r * torch.cos(th), r * torch.sin(th)


def _normals(seed, t, i, purpose, sub, n):
    """n standard normals of every (i, sub); a last axis of n."""
    out = []
    for b in range((n + 3) // 4):
        w = _philox(seed, t, i, purpose, sub, torch.full_like(i, b))
        out += [*_pair(w[0], w[1]), *_pair(w[2], w[3])]
    return torch.stack(out[:n], -1)


def _la_z(seed, t, i, k, n):
    """The look-ahead's common inner normals: with n <= 2, two inner particles a block."""
    if n > 2:
        return _normals(seed, t, i, LA_Z, k, n)
    w = _philox(seed, t, i, LA_Z, k >> 1, torch.zeros_like(i))
    odd = (k & 1).bool().expand_as(w[0])
    a, b = _pair(torch.where(odd, w[2], w[0]), torch.where(odd, w[3], w[1]))
    return torch.stack([a, b][:n], -1)


class _Clg:
    """The conditionally linear-Gaussian family, in the x-first order of its descriptor."""

    def __init__(self, spec):
        f = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
        d1, self.dy = spec.d1, spec.dy
        self.d1, self.d2 = d1, spec.d - d1
        A, Q, H, P0 = spec.A, spec.Q, spec.H, spec.P0
        self.Axx, self.Axz, self.Azx, self.Azz = f(A[:d1, :d1]), f(A[:d1, d1:]), f(A[d1:, :d1]), f(A[d1:, d1:])
        self.Hx, self.Hz = f(H[:, :d1]), f(H[:, d1:])
        self.Lqx, self.Lqz = f(np.linalg.cholesky(Q[:d1, :d1])), f(np.linalg.cholesky(Q[d1:, d1:]))
        self.LrInv = f(np.linalg.inv(np.linalg.cholesky(spec.R)))
        self.LqxInv = f(np.linalg.inv(np.linalg.cholesky(Q[:d1, :d1])))
        S = H[:, d1:] @ Q[d1:, d1:] @ H[:, d1:].T
        self.Ls, self.K = f(np.linalg.cholesky(S)), f(Q[d1:, d1:] @ H[:, d1:].T @ np.linalg.inv(S))
        self.lognorm = -0.5 * self.dy * math.log(2 * math.pi) - 0.5 * np.linalg.slogdet(spec.R)[1]
        G0 = P0[d1:, :d1] @ np.linalg.inv(P0[:d1, :d1])
        self.m0x, self.m0z, self.G0 = f(spec.m0[:d1]), f(spec.m0[d1:]), f(G0)
        self.Lp0x = f(np.linalg.cholesky(P0[:d1, :d1]))
        self.Lp0c = f(np.linalg.cholesky(P0[d1:, d1:] - G0 @ P0[:d1, d1:]))
        self.growth, self.qc, self.xz = spec.growth, spec.qc, bool(np.any(A[:d1, d1:]))

    def init(self, seed, i, M):
        z0 = torch.zeros_like(i)
        x = self.m0x + _normals(seed, 0, i, INIT_X, z0, self.d1) @ self.Lp0x.T
        j = torch.arange(M, device="cuda")
        e = _normals(seed, 0, i[:, None].expand(-1, M), INIT_Z, j[None, :], self.d2)
        return x, self.m0z + ((x - self.m0x) @ self.G0.T)[:, None, :] + e @ self.Lp0c.T

    def fx(self, x, z):
        m = x @ self.Axx.T
        if self.growth is not None:  # the source step of the first transition is 0
            a, b, c, _ = self.growth
            m = m + a * x + b * x / (1 + x * x) + c
        return m + z @ self.Axz.T

    def fz(self, x, z):
        return x @ self.Azx.T + z @ self.Azz.T

    def hx(self, x):
        h = x @ self.Hx.T
        return h if self.qc is None else h + self.qc * x * x

    def log_py(self, r):
        return self.lognorm - 0.5 * (r @ self.LrInv.T).square().sum(-1)


def _lookahead_clg(m, seed, y, i, M, L):
    """lw, the x part and the z part of the group's mean, of outer particles i at step 1."""
    x, z = m.init(seed, i, M)
    n, dr = len(i), torch.arange(L, device="cuda")
    iL, iM = i[:, None].expand(-1, L), i[:, None].expand(-1, M)
    j = (_philox(seed, 1, iL, LA_J, dr[None, :], torch.zeros_like(iL))[0] * M) >> 32  # equal weights
    zj = torch.gather(z, 1, j[..., None].expand(-1, -1, m.d2))
    xL = x[:, None, :].expand(-1, L, -1)
    xbb = m.fx(xL, zj) + _normals(seed, 1, iL, LA_X, dr[None, :], m.d1) @ m.Lqx.T
    fz = m.fz(x[:, None, :], z)
    v = _la_z(seed, 1, iM, torch.arange(M, device="cuda")[None, :], m.dy) @ m.Ls.T
    p = fz @ m.Hz.T + v
    res = ((y - m.hx(xbb)) @ m.LrInv.T)[:, :, None, :] - (p @ m.LrInv.T)[:, None, :, :]
    ell = m.lognorm - 0.5 * res.square().sum(-1)  # (n, L, M)
    alpha = torch.full((n, L, M), -math.log(M), dtype=torch.float64, device="cuda")
    if m.xz:
        fk = m.fx(x[:, None, :].expand(-1, M, -1), z)
        alpha = alpha - 0.5 * ((xbb[:, :, None, :] - fk[:, None, :, :]) @ m.LqxInv.T).square().sum(-1)
    top = torch.logsumexp(alpha + ell, 2)
    lwh = top - torch.logsumexp(alpha, 2)
    lw = torch.logsumexp(lwh, 1) - math.log(L)
    pi = torch.softmax(lwh, 1)
    beta = (torch.exp(alpha + ell - top[..., None]) * pi[..., None]).sum(1)  # (n, M)
    return lw, (pi[..., None] * xbb).sum(1), (beta[..., None] * (fz + v @ m.K.T)).sum(1)


def _particles_clg(m, seed, y, i):
    """The bootstrap filter's particles at step 1."""
    x, z = m.init(seed, i, 1)
    z = z[:, 0]
    s0 = torch.zeros_like(i)
    xn = m.fx(x, z) + _normals(seed, 1, i, PF_X, s0, m.d1) @ m.Lqx.T
    zn = m.fz(x, z) + _normals(seed, 1, i, PF_Z, s0, m.d2) @ m.Lqz.T
    return m.log_py(y - m.hx(xn) - zn @ m.Hz.T), xn, zn


def _standard_clg(m, seed, y, i, M):
    """The filter without look-ahead at step 1 (an x transition free of z: the local resampling
    then takes equal weights)."""
    x, z = m.init(seed, i, M)
    s0 = torch.zeros_like(i)
    xt = m.fx(x, z[:, 0]) + _normals(seed, 1, i, LA_X, s0, m.d1) @ m.Lqx.T
    iM, j = i[:, None].expand(-1, M), torch.arange(M, device="cuda")[None, :]
    zt = m.fz(x[:, None, :], z) + _normals(seed, 1, iM, PROP, j, m.d2) @ m.Lqz.T
    ell = m.log_py(y - m.hx(xt)[:, None, :] - zt @ m.Hz.T)
    lse = torch.logsumexp(ell, 1)
    return lse - math.log(M), xt, (torch.exp(ell - lse[:, None])[..., None] * zt).sum(1)


def _lookahead_paper(kind, seed, y, i, M, L):
    """The paper's models 1 and 2 at step 1 (source step 0): the inner draw given each x draw."""
    d = kind
    x = _normals(seed, 0, i, INIT_X, torch.zeros_like(i), d)
    iL, iM = i[:, None].expand(-1, L), i[:, None].expand(-1, M)
    k, dr = torch.arange(M, device="cuda")[None, :], torch.arange(L, device="cuda")[None, :]
    z = _normals(seed, 0, iM, INIT_Z, k, d)
    xk = x[:, None, :].expand(-1, M, -1)
    e = _la_z(seed, 1, iM, k, d)
    if kind == 1:
        fx = xk + z / (1 + z * z)
        fz = xk + 0.5 * z + 25 * z / (1 + z * z) + 8.0
        G, base = 0.1, math.sqrt(1 - 0.01) * e
    else:
        fx = torch.stack([0.5 * xk[..., 0], 0.4 * xk[..., 0] + 0.5 * xk[..., 1]], -1)
        q = z[..., 1] / (1 + z[..., 1] ** 2)
        z1 = z[..., 0] + q
        fz = torch.stack([z1, z1 + 0.5 * z[..., 1] + 25 * q + 8.0], -1)
        G, base = 0.0, torch.stack([e[..., 0], 1.1 * e[..., 0] + math.sqrt(11.2 - 1.21) * e[..., 1]], -1)
    j = (_philox(seed, 1, iL, LA_J, dr, torch.zeros_like(iL))[0] * M) >> 32
    xbb = torch.gather(fx, 1, j[..., None].expand(-1, -1, d)) + _normals(seed, 1, iL, LA_X, dr, d)
    dev = xbb[:, :, None, :] - fx[:, None, :, :]
    zh = (fz + base)[:, None, :, :] + G * dev  # (n, L, M, d)
    alpha = -math.log(M) - 0.5 * dev.square().sum(-1)
    if kind == 1:
        h = torch.atan(xbb[..., 0])[:, :, None] + zh[..., 0] ** 2 / 20
    else:
        h = ((xbb[..., 0] + xbb[..., 1]) / (1 + xbb[..., 0] ** 2))[:, :, None] + torch.atan(zh[..., 0]) + zh[..., 1] ** 2 / 20
    a1 = alpha - 0.5 * math.log(2 * math.pi) - 0.5 * (y - h) ** 2
    top = torch.logsumexp(a1, 2)
    lwh = top - torch.logsumexp(alpha, 2)
    pi = torch.softmax(lwh, 1)
    zrow = (torch.exp(a1 - top[..., None])[..., None] * zh).sum(2)
    return torch.logsumexp(lwh, 1) - math.log(L), (pi[..., None] * xbb).sum(1), (pi[..., None] * zrow).sum(1)


def _estimate(N, rows, part):
    """The filtered mean and the evidence from part(i) over outer particles in chunks of rows."""
    got = [part(torch.arange(a, min(N, a + rows), device="cuda")) for a in range(0, N, rows)]
    lw, s = torch.cat([g[0] for g in got]), torch.cat([torch.cat(g[1:], 1) for g in got])
    mx = lw.max()
    W = torch.exp(lw - mx)
    return (W @ s / W.sum()).cpu().numpy(), float(mx + torch.log(W.mean()))


def _lookahead_estimate(spec, N, M, L, seed, y):
    m = _Clg(spec)
    y = torch.as_tensor(y, dtype=torch.float64, device="cuda")
    rows = max(1, int(4e7 / (M * (L * (m.dy + (m.d1 if m.xz else 0)) + 2 * m.d2))))
    return _estimate(N, rows, lambda i: _lookahead_clg(m, seed, y, i, M, L))


def _network(W, F):
    a = F
    for q in (1, 2, 3):
        a = torch.relu(a @ W[f"W{q}"].T + W[f"b{q}"])
    return a @ W["W4"].T + W["b4"]


def _gradient(case, seed):
    form = case["form"]
    d1, d2, dy, din, dout = _proposal_shape(form)
    W = {k: torch.as_tensor(v, device="cuda").requires_grad_() for k, v in _proposal_weights(form, seed).items()}
    F, Z, w = (t.cuda().double() for t in _proposal_rows(case, seed))
    o = _network(W, F)
    if form == "wide":
        ls, c = o[:, :d2].clamp(-7, 5), o[:, d2:]
        zt, mu, k = Z[:, :d2], Z[:, d2:2 * d2], Z[:, 2 * d2:]
        r = k + (zt - k - c) * torch.exp(-ls) - mu
        nll = 0.5 * (r * r / 0.1).sum(1) + ls.sum(1) + 0.5 * d2 * math.log(2 * math.pi * 0.1)
    else:
        C = 4
        mu, ls = o[:, C:C + C * d2].reshape(-1, C, d2), o[:, C + C * d2:].clamp(-7, 5).reshape(-1, C, d2)
        q = (-0.5 * ((Z[:, None, :] - mu) * torch.exp(-ls)) ** 2 - ls - 0.5 * math.log(2 * math.pi)).sum(2)
        nll = -torch.logsumexp(torch.log_softmax(o[:, :C], 1) + q, 1)
    loss = (w * nll).sum() / w.sum()
    loss.backward()
    return {"loss": float(loss), "grad": torch.cat([W[f"{a}{q}"].grad.reshape(-1) for q in (1, 2, 3, 4) for a in "Wb"])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "resample":
        return None  # indices: whole numbers
    if kind == "grad":
        return _gradient(case, seed)
    if kind == "forward":
        W = {k: torch.as_tensor(v, device="cuda") for k, v in _proposal_weights("mixture", seed).items()}
        return {"head": _network(W, _proposal_rows(case, seed)[0].cuda().double())}
    if kind in ("online", "ladpf", "learned"):
        spec = _spec(case, seed)
        dt = np.float64 if kind == "online" else np.float32
        T = T_LINEAR if spec.growth is None else T_GROWTH
        y = workloads.simulate(spec, T, seed)[1][0].astype(dt)
        mean, lz = _lookahead_estimate(spec, case["N"], case["M"], case["L"], seed, y)
        return {"mean": mean, "logz": lz if kind == "online" else np.array([lz])}
    if kind == "batch":
        d1s, Ns, Ms, specs, seeds = _batch_members(case, seed)
        got = [_lookahead_estimate(s, Ns[f], Ms[f], case["L"], seeds[f], workloads.simulate(s, 128, seed + f)[1][0].astype(np.float32))
               for f, s in enumerate(specs)]
        return {"mean": np.concatenate([g[0] for g in got]), "logz": np.array([g[1] for g in got])}
    if kind == "paper":
        y = float(workloads.simulate_paper(case["model"], T_PAPER, seed)[1][0].astype(np.float32)[0])
        rows = max(1, int(4e7 / (case["M"] * case["L"] * 2 * case["model"])))
        mean, lz = _estimate(case["N"], rows, lambda i: _lookahead_paper(case["model"], seed, y, i, case["M"], case["L"]))
        return {"mean": mean, "logz": np.array([lz])}
    spec = _spec(case, seed)
    m = _Clg(spec)
    y = torch.as_tensor(_observations(spec, seed, np.float32)[0], dtype=torch.float64, device="cuda")
    if kind == "pf":
        mean, lz = _estimate(case["N"], 1 << 20, lambda i: _particles_clg(m, seed, y, i))
    elif m.xz:
        return None  # the first step already resamples by unequal weights: decided by FP32 roundings
    else:
        mean, lz = _estimate(case["N"], max(1, (1 << 22) // (case["M"] * m.d2)), lambda i: _standard_clg(m, seed, y, i, case["M"]))
    return {"mean": mean, "logz": np.array([lz])}
