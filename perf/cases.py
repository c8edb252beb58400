"""What a user has this library do, as cases that can be timed and compared.

Four kinds of work, each through the public binding (``paper_2310_07486_gb300.qsg``):

  step      the elementary step of a simulation: `sweeps` checkerboard sweeps of
            every configuration and one tempering step over the k ladder; the
            spins come back in a device tensor (the state a program checkpoints)
  measure   one measurement of C(tau), Q2(tau) and the one-time sums, finished
            in FP64 and read into page-locked host buffers
  monitor   a short step followed by a measurement and the reads of a program
            that follows a run (energies, overlaps or correlators)
  train / predict   the k-ladder predictor: Adam steps on mini-batches of host
            data, and inference on host features
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2310_07486_gb300 import qsg as Q
from paper_2310_07486_gb300 import workloads as W

# the rows of the ragged workload: (L, L_tau, ladder length, k_min, k_max)
RAGGED = [(8, 128, 16, 0.265, 0.305), (12, 256, 24, 0.265, 0.305), (16, 512, 48, 0.265, 0.295986),
          (20, 1024, 56, 0.265, 0.295986), (24, 2048, 60, 0.265, 0.292)]


def _case(name, kind, L, Ltau, samples, R, K, algo, boundary, k_min, k_max, **more):
    return dict(name=name, kind=kind, L=L, Ltau=Ltau, samples=samples, R=R, K=K, algo=algo, boundary=boundary,
                k_min=k_min, k_max=k_max, **more)


def listed():
    return [
        # the smallest run: one sample, two replicas at one k, measured every
        # 10 sweeps and read each time; launches and latency are all there is
        _case("monitor_L6_Lt32_one_sample", "monitor", 6, 32, 1, 2, 1, "metropolis", "pbc", 0.29, 0.29, sweeps=10,
              groups=1, graph=False, read="correlators"),
        # a training run of the k-ladder study: 640 samples at its middle size
        _case("monitor_L8_Lt48_640_samples", "monitor", 8, 48, 640, 4, 32, "heatbath", "pbc", 0.2, 0.45, sweeps=8,
              groups=1, graph=True, read="energies"),
        # the study's evaluation run: four groups of 64 samples, each on its
        # own ladder, one sweep graph over all groups
        _case("monitor_L12_Lt64_4_ladders", "monitor", 12, 64, 64, 4, 32, "heatbath", "pbc", 0.2, 0.45, sweeps=8,
              groups=4, graph=True, read="energies"),
        # the mid-scale workload (24 k in [0.20, 0.40], swaps every 10 sweeps),
        # launched directly
        _case("step_L16_Lt512_metropolis", "step", 16, 512, 64, 4, 24, "metropolis", "pbc", 0.20, 0.40, sweeps=10,
              graph=False),
        # an extent of tau that is no multiple of 16, antiperiodic, with a
        # partly filled last word of samples
        _case("step_L10_Lt200_antiperiodic", "step", 10, 200, 100, 4, 16, "metropolis", "apbc", 0.22, 0.36, sweeps=30,
              graph=False),
        # a lattice size between those of the simulation table
        _case("step_L18_Lt1024_heatbath", "step", 18, 1024, 64, 4, 16, "heatbath", "pbc", 0.22, 0.36, sweeps=30,
              graph=True),
        # the headline workload's elementary step: 30 sweeps and one tempering
        # step of 128 samples x 4 replicas x 32 k, 2.4 GB of spins
        _case("step_L24_Lt2048_heatbath", "step", 24, 2048, 128, 4, 32, "heatbath", "pbc", 0.22, 0.36, sweeps=30,
              graph=True),
        # 640 samples of five sizes in one context, 6.5 GB of spins
        dict(name="step_ragged_640", kind="step", ragged=True, sweeps=30, graph=True, algo="metropolis",
             boundary="pbc", samples=128, R=4),
        # the measurement of the headline lattice, at a quarter of its ladder
        # and one word of samples
        _case("measure_L24_Lt2048", "measure", 24, 2048, 64, 4, 8, "heatbath", "pbc", 0.22, 0.36),
        # a smaller lattice with six replicas (20 replica triples), antiperiodic
        _case("measure_L16_Lt512_6_replicas", "measure", 16, 512, 64, 6, 16, "metropolis", "apbc", 0.265, 0.295986),
        # one epoch of the predictor's training: 1920 samples, batches of 128
        dict(name="train_1920_batch128", kind="train", n=1920, batch=128, steps=15),
        # predicted ladders of 256 fresh samples
        dict(name="predict_256_bf16", kind="predict", n=256, bf16=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["measure"] * 3 + ["monitor"] * 2 + ["train", "predict"])
    if kind == "train":
        return dict(kind=kind, n=_log_int(rng, 256, 4096), batch=_log_int(rng, 16, 256), steps=_log_int(rng, 4, 48))
    if kind == "predict":
        return dict(kind=kind, n=_log_int(rng, 16, 4096), bf16=rng.random() < 0.7)
    small = kind == "monitor"
    L = 2 * rng.randint(3, 6 if small else 12)
    Ltau = _log_int(rng, 32, 128 if small else 2048)
    # most programs take a multiple of 16 (L_tau >= 32), the rest any even extent
    Ltau = max(32, Ltau // 16 * 16) if rng.random() < 0.75 else max(32, Ltau // 2 * 2)
    R = rng.choice([2, 3, 4, 4, 4, 6])
    samples = _log_int(rng, 1, 640 if small else 256)
    K = _log_int(rng, 1, 40 if small else 60)
    k_min = rng.uniform(0.2, 0.28)
    c = dict(kind=kind, L=L, Ltau=Ltau, R=R, algo=rng.choice(["metropolis", "heatbath"]),
             boundary=rng.choice(["pbc", "pbc", "apbc"]), k_min=k_min, k_max=k_min + rng.uniform(0.02, 0.15))
    words = lambda: (samples + 63) // 64 * R * K * L * L * Ltau  # noqa: E731
    if kind == "measure":
        # at most the sample bits and Gram elements of the largest listed measurement
        while (samples + 63) // 64 * 64 * R * K * float(Ltau) ** 2 * L * L > 64 * 4 * 8 * 2048.0 ** 2 * 576 \
                or (samples + 63) // 64 * 64 * K * Ltau * R ** 2 > 64 * 8 * 2048 * 36:
            samples, K = max(1, samples // 2), max(1, K * 2 // 3)
    else:
        c["sweeps"] = rng.choice([8, 10, 30])
        c["graph"] = Ltau % 16 == 0 and rng.random() < 0.6
        while words() > 3.0e8:
            samples, K = max(1, samples // 2), max(1, K * 2 // 3)
    if small:
        c["groups"] = rng.choice([1, 1, 2, 4])
        c["read"] = rng.choice(["energies", "energies", "correlators"])
    c.update(samples=samples, K=K)
    return c


# ---- inputs -----------------------------------------------------------------
def _shapes(c):
    algo = Q.METROPOLIS if c["algo"] == "metropolis" else Q.HEATBATH
    boundary = Q.PBC if c["boundary"] == "pbc" else Q.APBC
    if c.get("ragged"):
        return ([Q.Shape(L, Lt, c["samples"], c["R"], K, algo, boundary) for L, Lt, K, _, _ in RAGGED],
                [W.uniform_ladder(a, b, K) for _, _, K, a, b in RAGGED])
    n = c.get("groups", 1)
    # several groups stand for groups of samples on ladders of their own
    return ([Q.Shape(c["L"], c["Ltau"], c["samples"], c["R"], c["K"], algo, boundary) for _ in range(n)],
            [W.uniform_ladder(c["k_min"], c["k_max"] + 0.01 * g, c["K"]) for g in range(n)])


def spin_words(c, seed):
    """Spins of a measurement, int64 words [W][R][K][L_tau][L*L]: per sample and
    k one pattern in which an eighth of the spins flip from one slice to the
    next (a decay along tau), and in every replica an eighth of it flipped (an
    overlap between the replicas)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    Wn, n, Lt = (c["samples"] + 63) // 64, c["L"] ** 2, c["Ltau"]

    def words(*shape):
        return torch.randint(-2 ** 63, 2 ** 63 - 1, shape, dtype=torch.int64, device="cuda", generator=g)

    def eighth(*shape):
        return words(*shape) & words(*shape) & words(*shape)

    s = eighth(Wn, 1, c["K"], Lt, n)
    s[:, :, :, 0] = words(Wn, 1, c["K"], n)
    k = 1
    while k < Lt:  # running exclusive-or along tau
        s[:, :, :, k:] ^= s[:, :, :, :-k].clone()
        k *= 2
    return s ^ eighth(Wn, c["R"], c["K"], Lt, n)


def _mlp_inputs(c, seed):
    rng = np.random.default_rng(seed)
    X = rng.random((c["n"], 64), dtype=np.float32)  # fractions of lattice sites, as the coupling features are
    T = np.empty((c["n"], 33), dtype=np.float32)
    f = rng.gamma(4.0, size=(c["n"], 32))
    T[:, :32] = f / f.sum(axis=1, keepdims=True)
    T[:, 32] = rng.uniform(0.6, 0.9, c["n"])
    parts = []
    for shape in [(128, 64), (128,), (128, 128), (128,), (33, 128), (33,)]:
        lim = math.sqrt(6.0 / shape[1]) if len(shape) == 2 else 0.0
        parts.append(rng.uniform(-lim, lim, size=shape).ravel())
    theta = np.concatenate(parts).astype(np.float32)
    idx = rng.integers(0, c["n"], size=(c.get("steps", 1), c.get("batch", 1))).astype(np.int32)
    return X, T, theta, idx


def prepare(case, seed):
    c = dict(case)
    if c["kind"] in ("train", "predict"):
        X, T, theta, idx = _mlp_inputs(c, seed)
        m = Q.MLP(max(c["n"], 1024), c.get("batch", 128))
        m.set_params(theta)
        m.set_data(X, T)
        return dict(case=c, mlp=m, X=X, idx=idx)
    shapes, ladders = _shapes(c)
    ctx = Q.Context(shapes)
    ctx.qsg_init_samples(seed, ladders)
    state = dict(case=c, ctx=ctx, shapes=shapes)
    if c["kind"] == "measure":
        ctx.qsg_set_spins_device(0, spin_words(c, seed).reshape(-1))
        state["out"] = ctx.correlator_buffers(0, pinned=True)
        torch.cuda.synchronize()
        return state
    if c["kind"] == "monitor":
        for g, s in enumerate(shapes):
            ctx.qsg_set_couplings(g, W.bimodal_couplings(s.n_samples, s.L, seed + g))
        if c["read"] == "correlators":
            state["out"] = [ctx.correlator_buffers(g, pinned=True) for g in range(len(shapes))]
    if c["graph"]:
        ctx.qsg_set_option(Q.OPT_GRAPH, c["sweeps"])
    # away from the hot start, so that tempering meets ordinary energies
    ctx.qsg_sweep(5)
    if c["kind"] == "step":
        state["spins"] = [torch.empty(s.slots * s.Ltau * s.L * s.L, dtype=torch.int64, device=ctx.device)
                          for s in shapes]
    return state


def run(state):
    c = state["case"]
    if c["kind"] == "train":
        losses = state["mlp"].train(state["idx"], 2e-3)
        return dict(losses=losses, params=state["mlp"].get_params())
    if c["kind"] == "predict":
        return state["mlp"].predict(state["X"], bf16=c["bf16"])
    ctx, shapes = state["ctx"], state["shapes"]
    if c["kind"] == "measure":
        ctx.qsg_measure_correlators()
        out = dict(ctx.qsg_read_correlators(0, out=state["out"]))
        one = ctx.qsg_read_onetime(0)
        out.update(per_k=one.pop("per_k"), sums=one.pop("raw"), per_sample=one)
        return out
    ctx.qsg_sweep(c["sweeps"])
    ctx.qsg_tempering_swap()
    if c["kind"] == "step":
        for g, t in enumerate(state["spins"]):
            ctx.qsg_get_spins_device(g, t)
        return state["spins"]
    ctx.qsg_measure_correlators()
    if c["read"] == "correlators":
        return [ctx.qsg_read_correlators(g, out=state["out"][g]) for g in range(len(shapes))]
    return [[ctx.qsg_read_energies(g), ctx.qsg_read_pair_overlaps(g)] for g in range(len(shapes))]


# ---- the work a pass cannot do without -----------------------------------------
def _correlator_work(s):
    """Bytes and flops of one measurement: the spins read and the sums written
    once; a product and a sum per site of every pair of slices up to lag
    L_tau / 2."""
    bits = s.n_samples * s.n_replicas * s.n_k
    return 8.0 * s.slots * s.Ltau * s.L ** 2 + 16.0 * bits * s.n_lag, 2.0 * bits * s.Ltau * s.n_lag * s.L ** 2


def work(case):
    c = dict(case)
    params = 29089
    if c["kind"] == "train":
        B = c["batch"]
        return {"bytes": 4.0 * (6 * params + c["steps"] * B * 98), "flops": 6.0 * c["steps"] * B * params}
    if c["kind"] == "predict":
        return {"bytes": 4.0 * (params + c["n"] * 97), "flops": 2.0 * c["n"] * params}
    shapes, _ = _shapes(c)
    bytes_, flops = 0.0, 0.0
    for s in shapes:
        words = s.slots * s.Ltau * s.L ** 2
        if c["kind"] == "measure":
            b, f = _correlator_work(s)
            bytes_ += b
            flops += f
            continue
        # the state read and written once; an operation for each attempted
        # spin update (integer logic on words of 64 spins, not tensor work)
        bytes_ += 16.0 * words
        flops += 64.0 * words * c["sweeps"]
        if c["kind"] == "monitor":
            flops += _correlator_work(s)[1]
        else:
            bytes_ += 8.0 * words  # the copy that comes back
    return {"bytes": bytes_, "flops": flops}


# ---- the same results in 64 bits, without the library -----------------------------
def _exact_measure(c, seed):
    words = spin_words(c, seed)
    R, K, L, Lt, ns = c["R"], c["K"], c["L"], c["Ltau"], c["samples"]
    half, N = Lt // 2, L * L
    z = -1.0 if c["boundary"] == "apbc" else 1.0
    dev = words.device
    C = torch.zeros(R, ns, K, half + 1, dtype=torch.float64, device=dev)
    Q2 = torch.zeros_like(C)
    names = ("q2", "q4", "chi2", "F2", "chi3", "F3", "chi_lin")
    ps = torch.zeros(ns, K, len(names), dtype=torch.float64, device=dev)
    phase = torch.exp(2j * math.pi * torch.arange(L, device=dev, dtype=torch.float64) / L)
    pairs = [(a, b) for a in range(R) for b in range(a + 1, R)]
    triples = [(a, b, d) for a in range(R) for b in range(a + 1, R) for d in range(b + 1, R)]
    has3 = 3 <= R <= 8
    for i in range(ns):
        S = (1 - 2 * ((words[i // 64] >> (i % 64)) & 1)).to(torch.float32)  # [R][K][Lt][N]
        for r in range(R):
            ext = torch.cat([S[r], z * S[r][:, :half]], dim=1)
            G = torch.bmm(S[r], ext.transpose(1, 2).contiguous())
            D = G.as_strided((K, Lt, half + 1), (Lt * (Lt + half), Lt + half + 1, 1)).double()
            C[r, i] = D.sum(dim=1) / (N * Lt)
            Q2[r, i] = (D * D).sum(dim=1) / (float(N) ** 2 * Lt)
        X = S.double().reshape(R, K, Lt, L, L)
        if pairs:
            q, h = {}, {}
            for a, b in pairs:
                o = X[a] * X[b]
                q[a, b] = o.sum(dim=(2, 3))
                h[a, b] = [(o.sum(dim=2).to(phase.dtype) * phase).sum(dim=2),
                           (o.sum(dim=3).to(phase.dtype) * phase).sum(dim=2)]
            P = sum((v ** 2).sum(dim=1) for v in q.values())
            P4 = sum((v ** 4).sum(dim=1) for v in q.values())
            F = sum(sum((x.abs() ** 2).sum(dim=1) for x in v) for v in h.values())
            n = len(pairs) * Lt
            ps[i, :, 0], ps[i, :, 1] = P / (n * float(N) ** 2), P4 / (n * float(N) ** 4)
            ps[i, :, 2], ps[i, :, 3] = P / (n * N), F / (2.0 * n * N)
        if has3:
            T, F3 = 0.0, 0.0
            for a, b, d in triples:
                ab, bd, ad = (a, b), (b, d), (a, d)
                T = T + (q[ab] * q[bd] * q[ad]).sum(dim=1)
                for u, v, w in ((ab, ad, bd), (ab, bd, ad), (ad, bd, ab)):
                    F3 = F3 + sum((q[w] * (x * y.conj()).real).sum(dim=1) for x, y in zip(h[u], h[v]))
            n = len(triples) * Lt
            ps[i, :, 4], ps[i, :, 5] = T / (n * N), F3 / (6.0 * n * N)
        Ci = C[:, i]
        ps[i, :, 6] = (Ci[..., 0] + 2.0 * Ci[..., 1:half].sum(dim=-1) + Ci[..., half]).mean(dim=0)
    if not has3:
        ps[..., 4:6] = math.nan
    m = ps.mean(dim=0)
    s2 = 2.0 * math.sin(math.pi / L)
    per_k = dict(chi2=m[:, 2], F2=m[:, 3], xi2=torch.sqrt(m[:, 2] / m[:, 3] - 1.0) / s2, chi3=m[:, 4], F3=m[:, 5],
                 xi3=torch.sqrt(m[:, 4] / m[:, 5] - 1.0) / s2, B=m[:, 1] / m[:, 0] ** 2, chi_lin=m[:, 6])
    return dict(C=C, Q2=Q2, q2=ps[..., 0].clone(), per_k=per_k, sums=None,
                per_sample={f: ps[..., j].clone() for j, f in enumerate(names)})


def _layers(theta):
    t = torch.as_tensor(theta, dtype=torch.float64)
    out, o = [], 0
    for shape in [(128, 64), (128,), (128, 128), (128,), (33, 128), (33,)]:
        n = math.prod(shape)
        out.append(t[o:o + n].reshape(shape).clone().requires_grad_(True))
        o += n
    return out


def _forward(p, X):
    h = torch.relu(X @ p[0].T + p[1])
    h = torch.relu(h @ p[2].T + p[3])
    return h @ p[4].T + p[5]


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "measure":
        return _exact_measure(c, seed)
    if c["kind"] == "predict":
        X, _, theta, _ = _mlp_inputs(c, seed)
        return _forward(_layers(theta), torch.as_tensor(X, dtype=torch.float64)).detach()
    if c["kind"] == "train":
        X, T, theta, idx = _mlp_inputs(c, seed)
        X, T, p = torch.as_tensor(X, dtype=torch.float64), torch.as_tensor(T, dtype=torch.float64), _layers(theta)
        m, v, losses = [torch.zeros_like(x) for x in p], [torch.zeros_like(x) for x in p], []
        for t, ix in enumerate(idx, start=1):
            ix = torch.as_tensor(ix, dtype=torch.int64)
            y = _forward(p, X[ix])
            ce = -(T[ix][:, :32] * torch.log_softmax(y[:, :32], dim=1)).sum(dim=1)
            loss = (ce + (y[:, 32] - T[ix][:, 32]) ** 2).mean()
            losses.append(loss.item())
            for x, g, a, b in zip(p, torch.autograd.grad(loss, p), m, v):
                a.mul_(0.9).add_(0.1 * g)
                b.mul_(0.999).add_(0.001 * g * g)
                x.data -= 2e-3 * (a / (1 - 0.9 ** t)) / (torch.sqrt(b / (1 - 0.999 ** t)) + 1e-8)
        return dict(losses=torch.tensor(losses, dtype=torch.float64),
                    params=torch.cat([x.detach().reshape(-1) for x in p]))
    return None  # spins, energies and overlaps are whole numbers
