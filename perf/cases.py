"""Performance cases: the calls a program that uses this library makes, over the range of sizes
it makes them in.

Seven kinds, all through the public entry points of the Python package:

  step      one iteration of coded gradient descent: chunk gradients with the loss, Algorithm 1
            for the realization's finished chunks, then encode, decode and update
  grads     chunk gradients of one parameter vector alone
  batched   chunk gradients of several parameter vectors at once (a learning-rate sweep)
  decode    the parameter server's decode of a batch of straggler patterns: plan, then apply
  mse       the error measures alone of a batch of patterns (the sweep over completion rates)
  transmit  what the workers send for a few patterns (Algorithm 1 and eq. 2) and its decode,
            under the cyclic order or under Algorithm 2's order of a regular assignment
  trigger   completion times and the encode-and-transmit trigger of simulated realizations
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2405_19509_gb300 as gc

_DEV = "cuda"


# ------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the 6-worker example: every call is a few microseconds, so launches and latency count
        dict(name="step_tiny", kind="step", N=6, delta=3, ell=2, d=64, n_c=32, loss="lsq", x="f32"),
        # the 20-worker logistic regression, one live iteration (168 MB of features)
        dict(name="step_logistic", kind="step", N=20, delta=4, ell=2, d=4096, n_c=512,
             loss="logistic", x="f32"),
        # real tables seldom have a power of two of columns or of rows per chunk (666 MB)
        dict(name="step_ragged", kind="step", N=50, delta=5, ell=3, d=10007, n_c=333,
             loss="logistic", x="f32"),
        # the largest pass over features: 8.6 GB of long bf16 rows
        dict(name="grads_wide_bf16", kind="grads", N=64, d=65536, n_c=1024, loss="lsq", x="bf16"),
        # the same features against 256 parameter vectors (two dense contractions)
        dict(name="batched_256", kind="batched", N=64, d=65536, n_c=1024, n_w=256, loss="lsq"),
        # a server's ordinary batch: many patterns of a small model (164 MB written)
        dict(name="decode_logistic", kind="decode", N=20, delta=4, ell=2, d=4096, npat=10000,
             psi="shifted_exp"),
        # the largest decode: 4,096 patterns of a million parameters (17 GB written)
        dict(name="decode_large", kind="decode", N=256, delta=16, ell=2, d=1 << 20, npat=4096,
             psi="frac_binom"),
        # four blocks a gradient: most patterns miss some copies, the decode is a contraction
        dict(name="decode_l4", kind="decode", N=256, delta=16, ell=4, d=1 << 20, npat=1024,
             psi="frac_binom"),
        # errors only, 100,000 patterns with few chunks finished
        dict(name="mse_sweep", kind="mse", N=64, delta=8, ell=2, d=65536, npat=100000, p=0.3),
        # what 256 workers send in one realization (1.07 GB of chunk gradients)
        dict(name="transmit_cyclic", kind="transmit", N=256, delta=16, ell=2, d=1 << 20, npat=1,
             order="cyclic"),
        # the same on a regular graph's assignment, a few realizations, odd length
        dict(name="transmit_regular", kind="transmit", N=200, delta=8, ell=3, d=262147, npat=4,
             order="regular"),
        # the completion-time simulation of 200 workers
        dict(name="trigger", kind="trigger", N=200, delta=8, ell=2, theta=0, alpha=6, nsim=100000,
             order="cyclic"),
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "grads", "batched", "decode", "decode", "mse", "transmit",
                       "transmit", "trigger"])
    if kind == "step":
        N = _log(rng, 6, 128)
        delta = rng.randint(3, min(8, N))
        d = _log(rng, 64, 16384)
        n_c = _log(rng, 32, max(33, min(2048, (1 << 31) // (N * d))))
        return dict(kind=kind, N=N, delta=delta, ell=rng.randint(1, 3), d=_even(rng, d, 4),
                    n_c=_even(rng, n_c, 4), loss=rng.choice(["lsq", "logistic"]), x="f32")
    if kind == "grads":
        x = rng.choice(["f32", "bf16"])
        N = _log(rng, 8, 128)
        d = _log(rng, 1024, 65536)
        n_c = _log(rng, 32, max(33, min(2048, (1 << (31 if x == "bf16" else 30)) // (N * d))))
        return dict(kind=kind, N=N, d=_even(rng, d, 8), n_c=_even(rng, n_c, 4),
                    loss=rng.choice(["lsq", "logistic"]), x=x)
    if kind == "batched":
        N = 2 * _log(rng, 4, 32)
        n_c = 64 * _log(rng, 2, 16)
        return dict(kind=kind, N=N, n_c=n_c, d=128 * _log(rng, 8, min(512, (1 << 24) // (N * n_c))),
                    n_w=32 * rng.randint(1, 8), loss=rng.choice(["lsq", "logistic"]))
    if kind == "decode":
        N = _log(rng, 20, 256)
        delta = rng.randint(4, 16)
        npat = _log(rng, 64, 10000)
        d = _log(rng, 4096, min(1 << 20, (1 << 31) // npat))
        return dict(kind=kind, N=N, delta=delta, ell=rng.randint(1, 4), d=_even(rng, d, 16),
                    npat=npat, psi=rng.choice(["shifted_exp", "frac_binom"]))
    if kind == "mse":
        return dict(kind=kind, N=_log(rng, 20, 80), delta=rng.randint(4, 10), ell=rng.randint(1, 3),
                    d=_even(rng, _log(rng, 4096, 65536), 8), npat=_log(rng, 1000, 100000),
                    p=rng.choice([0.3, 0.5, 0.7]))
    if kind == "transmit":
        N = _log(rng, 20, 256)
        order = rng.choice(["cyclic", "regular"])
        delta = rng.randint(4, 16) if order == "cyclic" else 2 * rng.randint(2, 5)
        npat = rng.randint(1, 8)
        return dict(kind=kind, N=N, delta=delta, ell=rng.randint(1, 4),
                    d=_even(rng, _log(rng, 4096, (1 << 20) // npat), 16), npat=npat, order=order)
    N = _log(rng, 50, 300)
    delta = 2 * rng.randint(2, 5)
    ell = rng.randint(1, 3)
    return dict(kind="trigger", N=N, delta=delta, ell=ell, theta=rng.choice([0, 0, N // 20]),
                alpha=rng.randint(0, delta - ell), nsim=_log(rng, 1000, 100000),
                order=rng.choice(["cyclic", "regular"]))


def _even(rng, n, q):
    """n as it is in half of the draws, else rounded up to a multiple of q."""
    return n if rng.random() < 0.5 else -(-n // q) * q


# ------------------------------------------------------------------------------------ inputs
def _gen(seed, tag):
    return torch.Generator(device=_DEV).manual_seed((seed * 1000003 + tag * 7919 + 12345) % (1 << 62))


def _randn(shape, g, dtype=torch.float32):
    return torch.randn(shape, generator=g, device=_DEV, dtype=dtype)


def _order(c, seed):
    """m x delta processing order on the host: cyclic, or Algorithm 2's order of a regular
    assignment (a circulant one with random offsets under random labels of chunks and workers)."""
    N, delta = c["N"], c["delta"]
    if c.get("order", "cyclic") == "cyclic":
        return gc.gc_make_assignment(N, N, delta, gc.GC_CYCLIC)[1]
    r = np.random.default_rng(seed)
    off, rows, cols = r.choice(N, size=delta, replace=False), r.permutation(N), r.permutation(N)
    A = np.zeros((N, N), dtype=np.uint8)
    for o in off:
        A[rows, cols[(np.arange(N) + o) % N]] = 1
    return gc.gc_chunk_ordering(A)[0]


def _patterns(model, npat, m, delta, g, p=None):
    """npat x m finished counts: shifted_exp (deadline when the slowest worker is half done),
    binomial (p), frac_binom (a completion rate per pattern, uniform in [0.2, 1])."""
    if model == "shifted_exp":
        tau = 1.0 + torch.empty(npat, m, device=_DEV, dtype=torch.float64).exponential_(generator=g)
        T = 0.5 * delta * tau.amax(1, keepdim=True)
        return torch.clamp(torch.floor(T / tau), max=delta).to(torch.int32).contiguous()
    f = torch.full((npat, 1, 1), p, device=_DEV) if p is not None else (
        0.2 + 0.8 * torch.rand(npat, 1, 1, generator=g, device=_DEV))
    u = torch.rand(npat, m, delta, generator=g, device=_DEV)
    return (u < f).sum(-1).to(torch.int32).contiguous()


def _features(c, g):
    """X, labels and the iterate.  The labels follow a generating vector with 256 non-zeros."""
    rows, d = c["N"] * c["n_c"], c["d"]
    bf16 = c.get("x", "bf16") == "bf16"
    X = _randn((rows, d), g, torch.bfloat16 if bf16 else torch.float32)
    if c["loss"] == "logistic" and not bf16:
        X.mul_(1.0 / math.sqrt(d))
    k = min(d, 256)
    z = (X[:, :k].float() * _randn((k,), g)).sum(1)
    if c["loss"] == "lsq":
        y = z / math.sqrt(k) + 0.1 * _randn((rows,), g)
    else:
        y = torch.where(torch.rand(rows, generator=g, device=_DEV) < torch.sigmoid(z), 1.0, -1.0)
    return X, y.float().contiguous()


def prepare(case, seed):
    c, kind = case, case["kind"]
    g = _gen(seed, 1)
    s = {"case": c, "ws": gc.Workspace(_DEV)}
    if kind in ("step", "grads", "batched"):
        s["X"], s["y"] = _features(c, g)
    if kind == "batched":
        s["W"] = _randn((c["n_w"], c["d"]), g) / math.sqrt(c["d"])
        s["G"] = torch.empty(c["n_w"], c["N"], c["d"], device=_DEV)
        return s
    if kind in ("step", "grads"):
        s["w"] = _randn((c["d"],), g) / math.sqrt(c["d"])
        s["G"] = torch.empty(c["N"], c["d"], device=_DEV)
        s["loss"] = torch.empty(1, device=_DEV, dtype=torch.float64)
        if kind == "grads":
            return s
    N = m = c["N"]
    ell, delta = c["ell"], c["delta"]
    s["order"] = torch.from_numpy(_order(c, seed)).to(_DEV)
    if kind == "trigger":
        tau = torch.empty(c["nsim"], m, device=_DEV, dtype=torch.float64).exponential_(generator=g)
        if c["alpha"]:
            dead = torch.rand(c["nsim"], m, generator=g, device=_DEV).topk(c["alpha"], 1).indices
            tau.scatter_(1, dead, math.inf)
        s["tau"] = tau
        f64 = dict(device=_DEV, dtype=torch.float64)
        s["T"], s["T_full"] = torch.empty(c["nsim"], **f64), torch.empty(c["nsim"], **f64)
        s["psi"] = torch.empty(c["nsim"], m, device=_DEV, dtype=torch.int32)
        return s
    s["R"] = _randn((ell, m), g, torch.float64)
    if kind == "step":
        s["psi"] = _patterns("shifted_exp", 1, m, delta, g)
        s["E"] = torch.empty(1, m, delta, ell, device=_DEV, dtype=torch.float64)
        s["w1"], s["ghat"] = torch.empty_like(s["w"]), torch.empty(c["d"], device=_DEV)
        return s
    npat, d = c["npat"], c["d"]
    s["G"] = _randn((N, d), g)
    if kind == "mse":
        s["psi"] = _patterns("binomial", npat, m, delta, g, c["p"])
    elif kind == "decode":
        s["psi"] = _patterns(c["psi"], npat, m, delta, g)
        s["plan"] = torch.empty(int(gc.lib.gc_decode_plan_bytes(N, ell, npat)), dtype=torch.uint8, device=_DEV)
        s["Ghat"] = torch.empty(npat, d, device=_DEV)
    else:
        s["psi"] = _patterns("frac_binom", npat, m, delta, g)
        s["T"] = torch.empty(npat, m, gc.block_length(d, ell), device=_DEV)
        s["ghat"] = torch.empty(npat, d, device=_DEV)
    if kind != "transmit":
        for k in ("coef_err", "est", "grad_mse"):
            s[k] = torch.empty(npat, device=_DEV, dtype=torch.float64)
    return s


_LOSS = {"lsq": gc.GC_LSQ, "logistic": gc.GC_LOGISTIC}
_LR = 0.5


def run(s):
    c = s["case"]
    kind, ws, N = c["kind"], s["ws"], c["N"]
    if kind == "batched":
        return {"G": gc.gc_chunk_grads_batched(s["X"], s["y"], s["W"], N, c["n_c"], _LOSS[c["loss"]],
                                               G=s["G"], ws=ws)}
    if kind in ("step", "grads"):
        gc.gc_chunk_grads(s["X"], s["y"], s["w"], N, c["n_c"], _LOSS[c["loss"]], G=s["G"],
                          loss_out=s["loss"], ws=ws)
        if kind == "grads":
            return {"G": s["G"], "loss": s["loss"]}
    ell, delta, m, order = c["ell"], c["delta"], N, s["order"]
    if kind == "trigger":
        return gc.gc_trigger_times(order, N, m, delta, s["tau"], ell, c["theta"], T=s["T"],
                                   psi=s["psi"], T_full=s["T_full"], ws=ws)
    R, psi, G = s["R"], s["psi"], s["G"]
    if kind == "step":
        gc.gc_find_encoding_coeff(R, ell, order, N, m, delta, psi, E=s["E"], C=False,
                                  delta_out=False, coef_err=False, est=False, ws=ws)
        s["w1"].copy_(s["w"])  # the step starts from the iterate it was handed
        gc.gc_live_step(s["E"], R, ell, order, N, m, delta, psi, G, s["w1"], _LR, N * c["n_c"],
                        ghat=s["ghat"])
        return {"G": G, "loss": s["loss"], "E": s["E"], "ghat": s["ghat"], "w": s["w1"]}
    if kind == "mse":
        return gc.gc_mse(R, ell, order, N, m, delta, psi, G, coef_err=s["coef_err"], est=s["est"],
                         grad_mse=s["grad_mse"], ws=ws)
    if kind == "decode":
        p = gc.gc_decode_plan(R, ell, order, N, m, delta, psi, plan=s["plan"],
                              coef_err=s["coef_err"], est=s["est"], ws=ws)
        r = gc.gc_decode_apply(p["plan"], ell, N, c["npat"], G, Ghat=s["Ghat"],
                               grad_mse=s["grad_mse"], ws=ws)
        return {"Ghat": r["Ghat"], "grad_mse": r["grad_mse"], "coef_err": p["coef_err"], "est": p["est"]}
    gc.gc_encode(R, ell, order, N, m, delta, psi, G, T=s["T"], ws=ws)
    gc.gc_decode_tx(R, ell, m, s["T"], c["d"], ghat=s["ghat"])
    return {"T": s["T"], "ghat": s["ghat"]}


# ------------------------------------------------------------------------------------ work
def work(case):
    c, kind, N = case, case["kind"], case["N"]
    if kind == "trigger":
        # every speed read once, every outcome written once; one product per (worker, slot)
        return {"bytes": c["nsim"] * (N * 8 + N * 4 + 16), "flops": 2.0 * c["nsim"] * N * c["delta"]}
    d = c["d"]
    if kind in ("step", "grads", "batched"):
        rows = N * c["n_c"]
        n_w = c.get("n_w", 1)
        by = rows * d * (2 if c.get("x", "bf16") == "bf16" else 4) + rows * 4 + n_w * d * 4 + n_w * N * d * 4
        fl = 4.0 * rows * d * n_w
        if kind == "step":
            by += N * d * 4 + 2 * d * 4 + N * c["delta"] * c["ell"] * 8
            fl += 2.0 * N * d * c["delta"] + 2.0 * N * d
        return {"bytes": by, "flops": fl}
    ell, delta, npat = c["ell"], c["delta"], c["npat"]
    by = N * d * 4 + npat * N * 4
    if kind == "transmit":
        L = -(-d // ell)
        # T goes out and comes in again: it is what crosses the network
        return {"bytes": by + 2 * npat * N * L * 4 + npat * d * 4,
                "flops": npat * (2.0 * N * delta * ell * L + 2.0 * N * ell * L)}
    # decoding writes each pattern's gradient; its sum over the chunks is shared by the batch
    return {"bytes": by + npat * (24 + (d * 4 if kind == "decode" else 0)), "flops": 1.0 * N * d}


# ------------------------------------------------------------------------------------ tolerances
def tolerance(case):
    # Errors against 64 bits measured over the listed cases and 150 drawn ones; the bounds are about
    # four times the largest seen.  2-norms: step 6e-7 (its decode up to 2e-5 where a block is ill
    # conditioned, as transmit's), grads 5e-7, batched 1.1e-4 (hi + lo bf16 products, long fp32
    # sums), decode 2.7e-6 (hi + lo bf16 products), mse 1.9e-6, transmit 1.7e-5.
    kind = case["kind"]
    if kind == "trigger":
        return "exact"  # every time is one product of a whole number and a double
    return {"step": {"rel": 2e-5, "max": 1e-3}, "grads": {"rel": 2.5e-6, "max": 2e-5},
            "batched": {"rel": 4.5e-4, "max": 2.5e-3}, "decode": {"rel": 1.1e-5, "max": 1e-4},
            "mse": {"rel": 8e-6, "max": 4e-5}, "transmit": {"rel": 8e-5, "max": 1e-3}}[kind]


# ------------------------------------------------------------------------------------ in 64 bits
def _exact_grads(s):
    """Chunk gradients and mean loss in 64 bits (as plain sums over each chunk's rows)."""
    c = s["case"]
    N, n_c = c["N"], c["n_c"]
    W = (s["W"] if c["kind"] == "batched" else s["w"][None]).double()
    G = torch.empty(W.shape[0], N, c["d"], device=_DEV, dtype=torch.float64)
    total = 0.0
    for i in range(N):
        x, y = s["X"][i * n_c:(i + 1) * n_c].double(), s["y"][i * n_c:(i + 1) * n_c, None].double()
        z = x @ W.T
        if c["loss"] == "lsq":
            r = z - y
            total = total + (0.5 * r * r)[:, 0].sum()
        else:
            r = torch.sigmoid(z) - 0.5 * (y + 1)
            total = total + torch.nn.functional.softplus(-y * z)[:, 0].sum()
        G[:, i] = r.T @ x
    return G, total / (N * n_c)


def _holders(order, N):
    """Worker and slot of every copy of every chunk (N x H, -1 past the last copy)."""
    lists = [[] for _ in range(N)]
    for j, row in enumerate(order.tolist()):
        for p, i in enumerate(row):
            lists[i].append((j, p))
    H = max(len(h) for h in lists)
    w = np.full((N, H), -1)
    p = np.zeros((N, H), dtype=np.int64)
    for i, h in enumerate(lists):
        for k, (a, b) in enumerate(sorted(h)):
            w[i, k], p[i, k] = a, b
    return w, p


def _have(s):
    """npat x N x H: which copies of every chunk are finished."""
    w, p = _holders(s["order"].cpu().numpy(), s["case"]["N"])
    w, p = torch.from_numpy(w).to(_DEV), torch.from_numpy(p).to(_DEV)
    return (s["psi"][:, w.clamp(min=0)] > p) & (w >= 0), w, p


def _pinv(s, chunk, have):
    """The pseudo-inverses (n x H x ell) of R restricted to the finished copies of `chunk`."""
    w = _holders(s["order"].cpu().numpy(), s["case"]["N"])[0]
    R = s["R"].cpu().numpy()
    X = R[:, np.maximum(w[chunk], 0)].transpose(1, 0, 2) * have[:, None, :]
    return np.linalg.pinv(X), X


def _coefficients(s):
    """E (npat x m x delta x ell) in 64 bits: Algorithm 1."""
    c = s["case"]
    N, m, delta, ell = c["N"], c["N"], c["delta"], c["ell"]
    have, w, p = (t.cpu().numpy() for t in _have(s))
    E = np.zeros((have.shape[0], m, delta, ell))
    for b in range(have.shape[0]):
        P = _pinv(s, np.arange(N), have[b])[0]
        i, h = np.nonzero(w >= 0)
        E[b, w[i, h], p[i, h]] = P[i, h]
    return torch.from_numpy(E).to(_DEV)


def _blocks(G, ell):
    """N x d gradients as N x ell x L blocks, the last one padded with zeros."""
    N, d = G.shape
    L = -(-d // ell)
    return torch.nn.functional.pad(G, (0, ell * L - d)).view(N, ell, L)


def _transmit(s, E, G):
    """T (npat x m x L) and its decode (npat x d) in 64 bits."""
    ell, d = s["case"]["ell"], G.shape[1]
    B = _blocks(G, ell)
    order = s["order"].long()
    T = torch.zeros(E.shape[0], order.shape[0], B.shape[2], device=_DEV, dtype=torch.float64)
    for p in range(order.shape[1]):
        for k in range(ell):
            T += E[:, :, p, k, None] * B[order[:, p], k]
    return T, torch.einsum("kj,bjc->bkc", s["R"], T).reshape(E.shape[0], -1)[:, :d]


def _departures(s):
    """Where a decode block differs from the identity (fewer than ell copies): pattern, chunk and
    the difference (n x ell x ell); with each pattern's coefficient error and estimate."""
    c = s["case"]
    N, ell = c["N"], c["ell"]
    have, _, _ = _have(s)
    missing = (ell - have.sum(-1)).clamp(min=0)
    b, i = torch.nonzero(missing, as_tuple=True)
    hv = have[b, i]
    H = hv.shape[1]
    key = i * (1 << H) + (hv.long() << torch.arange(H, device=_DEV)).sum(1)
    u, inv = torch.unique(key, return_inverse=True)
    u = u.cpu().numpy()
    mask = ((u[:, None] >> np.arange(H)) & 1).astype(bool)
    if len(u):
        P, X = _pinv(s, u >> H, mask)
        D = X @ P - np.eye(ell)
    else:
        D = np.zeros((0, ell, ell))
    D = torch.from_numpy(D).to(_DEV)[inv]
    npat = have.shape[0]
    ce = torch.zeros(npat, device=_DEV, dtype=torch.float64).index_add_(0, b, D.square().sum((1, 2)))
    return b, i, D, ce, missing.sum(1).double()


def _decode(s, keep):
    c = s["case"]
    N, ell, d, npat = c["N"], c["ell"], c["d"], c["npat"]
    b, i, D, ce, est = _departures(s)
    G = s["G"].double()
    full, B = G.sum(0), _blocks(G, ell)
    L = B.shape[2]
    B = B.reshape(N * ell, L)
    mse = torch.zeros(npat, device=_DEV, dtype=torch.float64)
    Ghat = full.repeat(npat, 1) if keep else None
    hit = torch.unique(b)
    step = max(1, (1 << 29) // (ell * L))
    for a in range(0, len(hit), step):
        rows = hit[a:a + step]
        at = torch.full((npat,), -1, device=_DEV, dtype=torch.long)
        at[rows] = torch.arange(len(rows), device=_DEV)
        sel = at[b] >= 0
        C = torch.zeros(len(rows), ell, N, ell, device=_DEV, dtype=torch.float64)
        C[at[b[sel]], :, i[sel], :] = D[sel]
        e = (C.view(len(rows) * ell, N * ell) @ B).view(len(rows), ell * L)[:, :d]
        mse[rows] = e.square().sum(1) / d
        if keep:
            Ghat[rows] += e
        del e, C
    return Ghat, mse, ce, est


def _trigger(s):
    c = s["case"]
    N, ell, delta = c["N"], c["ell"], c["delta"]
    w, p = _holders(s["order"].cpu().numpy(), N)
    w, p = torch.from_numpy(w).to(_DEV), torch.from_numpy(p).to(_DEV)
    T, F, S = [], [], []
    for tau in s["tau"].split(10000):
        def when(t):
            first = t.sort(-1).values[..., :ell].reshape(len(t), -1)
            return first.sort(-1).values[:, N * ell - 1 - c["theta"]] if c["theta"] < N * ell else t.new_zeros(len(t))
        t = when(tau[:, w] * (p + 1).double())
        T.append(t)
        F.append(when(tau[:, w] * float(delta)))
        done = (tau[:, :, None] * torch.arange(1, delta + 1, device=_DEV).double() <= t[:, None, None]).sum(-1)
        S.append(torch.where(torch.isinf(tau), 0, done).to(torch.int32))
    return {"T": torch.cat(T), "psi": torch.cat(S), "T_full": torch.cat(F)}


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "trigger":
        return _trigger(s)
    if kind in ("step", "grads", "batched"):
        G, loss = _exact_grads(s)
        if kind == "batched":
            return {"G": G}
        G, loss = G[0], loss.reshape(1)
        if kind == "grads":
            return {"G": G, "loss": loss}
        E = _coefficients(s)
        ghat = _transmit(s, E, G)[1][0]
        w = s["w"].double() - _LR * ghat / (case["N"] * case["n_c"])
        return {"G": G, "loss": loss, "E": E, "ghat": ghat, "w": w}
    if kind == "transmit":
        T, ghat = _transmit(s, _coefficients(s), s["G"].double())
        return {"T": T, "ghat": ghat}
    Ghat, mse, ce, est = _decode(s, kind == "decode")
    r = {"coef_err": ce, "est": est, "grad_mse": mse}
    return {**r, "Ghat": Ghat} if kind == "decode" else r
