"""Performance cases: the calls a user of this library makes, over the range
of sizes, dimensions, precisions and options they make them with.

Sizes and recipes are those of the repository's workloads, tests and benchmark
(``paper_1905_04582_gb300/workloads.py``): N = 200, the batch of 1600 / 1500 /
1300 / 992 items x 8 chains, the paper's 5392 items in four subtypes, the
sweep to N = 20000 and 50000 with D = 2 and 6; the others are generic and
ragged (no multiple of the 64-item block).  Locations come from a Gaussian
mixture (or N(0, I)), dissimilarities from the model, |distance + noise|, and
the evaluation point is the true one plus a jitter.

Kinds of a case:
  grad      new locations, then L, dL/dX and dL/dsigma from one fused pass
  autograd  the same through torch.autograd: forward and backward over (X, sigma)
  leapfrog  a leapfrog trajectory from new locations and momenta
  tree      the same with the phylogenetic prior in the target
  hmc       HMC iterations with the caller's draws (Metropolis included)
  batch     several datasets x chains: one HMC iteration of all chains
  cv        a cross-validation fold: training gradient, predictive density
  load      a new data set: Y into the library, then the first evaluation
  noalloc   the allocation-free FP64 entry point

Outputs of the FP32C path are returned in 32 bits (its arithmetic), those of
the FP64 paths in 64.  H(end) - H(start) is left out: a difference of two
energies of size 1e6, it holds only their rounding.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1905_04582_gb300 import capi
from paper_1905_04582_gb300.mds import MDS, Batch, mds_loglik

DEV = "cuda"


def listed():
    return [
        # the smallest call: an external sampler or optimiser evaluates a small
        # problem at new locations; latency, launches and waits are all of it
        {"name": "grad_n200_d2", "kind": "grad", "n": 200, "d": 2, "comps": 0, "sigma": 0.5, "prec": "fp32c",
         "order": False},
        # a whole small fit's inner loop: 10 iterations of 10 leapfrog steps
        {"name": "hmc_n200_d2", "kind": "hmc", "n": 200, "d": 2, "comps": 0, "sigma": 0.5, "iters": 10, "steps": 10,
         "eps": 1e-3},
        # the differentiable form at the paper's size, items in the caller's order
        {"name": "autograd_n5392_d2", "kind": "autograd", "n": 5392, "d": 2, "comps": 6, "sigma": 0.3, "order": False},
        # the paper's sampler step: 20 leapfrog steps at the paper's size, items in locality order
        {"name": "leapfrog_n5392_d2", "kind": "leapfrog", "n": 5392, "d": 2, "comps": 6, "sigma": 0.3, "order": True,
         "steps": 20, "eps": 1e-3},
        # the same with the paper's four subtype trees as the prior
        {"name": "tree_n5392_d2", "kind": "tree", "n": 5392, "d": 2, "sigma": 0.3, "order": True, "steps": 10,
         "eps": 1e-3, "trees": "1370,1389,1393,1240"},
        # six latent dimensions, a large problem
        {"name": "grad_n20000_d6", "kind": "grad", "n": 20000, "d": 6, "comps": 12, "sigma": 0.3, "prec": "fp32c",
         "order": True},
        # the largest: 1.25e9 pairs, 5 GB of Y
        {"name": "grad_n50000_d2", "kind": "grad", "n": 50000, "d": 2, "comps": 12, "sigma": 0.3, "prec": "fp32c",
         "order": True},
        # the FP64 context at the paper's size
        {"name": "grad_fp64_n5392_d2", "kind": "grad", "n": 5392, "d": 2, "comps": 6, "sigma": 0.3, "prec": "fp64",
         "order": False},
        # the FP64 entry point for callers that must not allocate; ragged N, padded rows, odd D
        {"name": "noalloc_n3001_d3", "kind": "noalloc", "n": 3001, "d": 3, "comps": 6, "sigma": 0.4, "pad": 7},
        # four datasets of uneven size, eight chains each, advanced together
        {"name": "batch_4x8_d2", "kind": "batch", "ns": "1600,1500,1300,992", "d": 2, "chains": 8, "comps": 6,
         "sigma": 0.3, "steps": 20, "eps": 5e-4},
        # model selection: a fold of 5 % held-out pairs, ragged N, three dimensions
        {"name": "cv_n2999_d3", "kind": "cv", "n": 2999, "d": 3, "comps": 6, "sigma": 0.4, "held": 0.05},
        # a new data set of 12000 items, full FP32 matrix on the device
        {"name": "load_n12000_d2", "kind": "load", "n": 12000, "d": 2, "comps": 12, "sigma": 0.3, "layout": "full",
         "y64": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grad", "grad", "grad", "grad64", "hmc", "autograd", "leapfrog", "leapfrog", "tree", "noalloc",
                       "batch", "cv", "load"])
    d = rng.choice([1, 2, 2, 2, 3, 4, 5, 6, 6, 7, 8])
    comps = rng.choice([0, 6, 12])
    sigma = rng.choice([0.2, 0.3, 0.4, 0.5])
    order = rng.random() < 0.5
    if kind == "grad":
        return {"kind": "grad", "n": _log_int(rng, 100, 24000), "d": d, "comps": comps, "sigma": sigma,
                "prec": "fp32c", "order": order}
    if kind == "grad64":
        return {"kind": "grad", "n": _log_int(rng, 100, 6000), "d": d, "comps": comps, "sigma": sigma, "prec": "fp64",
                "order": order}
    if kind == "hmc":
        return {"kind": "hmc", "n": _log_int(rng, 50, 800), "d": rng.choice([1, 2, 2, 3, 4, 6]), "comps": 0,
                "sigma": 0.5, "iters": rng.randint(2, 10), "steps": rng.randint(5, 20), "eps": 1e-3}
    if kind == "autograd":
        return {"kind": "autograd", "n": _log_int(rng, 100, 12000), "d": d, "comps": comps, "sigma": sigma,
                "order": order}
    if kind == "leapfrog":
        n = _log_int(rng, 300, 8000)
        return {"kind": "leapfrog", "n": n, "d": d, "comps": comps, "sigma": sigma, "order": order,
                "steps": rng.randint(5, 20), "eps": 0.07 / math.sqrt(n)}
    if kind == "tree":
        sizes = [_log_int(rng, 50, 1400) for _ in range(rng.randint(1, 4))]
        n = sum(sizes)
        return {"kind": "tree", "n": n, "d": rng.choice([1, 2, 2, 3, 4]), "sigma": sigma, "order": order,
                "steps": rng.randint(3, 10), "eps": 0.07 / math.sqrt(n), "trees": ",".join(str(s) for s in sizes)}
    if kind == "noalloc":
        return {"kind": "noalloc", "n": _log_int(rng, 50, 5000), "d": d, "comps": comps, "sigma": sigma,
                "pad": rng.randint(0, 9)}
    if kind == "batch":
        ns = [_log_int(rng, 300, 2000) for _ in range(rng.randint(2, 4))]
        return {"kind": "batch", "ns": ",".join(str(s) for s in ns), "d": rng.choice([1, 2, 2, 3, 4]),
                "chains": rng.randint(2, 8), "comps": 6, "sigma": sigma, "steps": rng.randint(5, 20), "eps": 5e-4}
    if kind == "cv":
        return {"kind": "cv", "n": _log_int(rng, 300, 6000), "d": d, "comps": comps, "sigma": sigma,
                "held": rng.choice([0.01, 0.05, 0.1])}
    return {"kind": "load", "n": _log_int(rng, 500, 14000), "d": rng.choice([2, 2, 3, 6]), "comps": comps,
            "sigma": sigma, "layout": rng.choice(["full", "packed"]), "y64": rng.random() < 0.3}


# ------------------------------------------------------------------ inputs


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _cloud(n, d, comps, g):
    """True locations: N(0, I), or a mixture with centres uniform in [-5, 5]^D, spread 0.3."""
    z = torch.randn(n, d, generator=g, device=DEV, dtype=torch.float64)
    if comps == 0:
        return z
    centres = 10.0 * torch.rand(comps, d, generator=g, device=DEV, dtype=torch.float64) - 5.0
    label = torch.randint(0, comps, (n,), generator=g, device=DEV)
    return centres[label] + 0.3 * z


def _dissimilarities(x, noise, g, ld=None):
    """Full N x N FP32 matrix (upper triangle meant) of |distance + noise|; rows of `ld` elements."""
    n, d = x.shape
    y = torch.zeros(n, ld or n, device=DEV, dtype=torch.float32)
    xf = x.float()
    block = max(64, min(n, (1 << 26) // n))
    for i0 in range(0, n, block):
        i1 = min(n, i0 + block)
        d2 = torch.zeros(i1 - i0, n - i0, device=DEV, dtype=torch.float32)
        for k in range(d):
            d2 += (xf[i0:i1, k, None] - xf[None, i0:, k]).square()
        d2.sqrt_()
        d2 += noise * torch.randn(i1 - i0, n - i0, generator=g, device=DEV, dtype=torch.float32)
        y[i0:i1, i0:n] = d2.abs_()
    return y


def _problem(n, d, comps, sigma, seed, ld=None):
    g = _gen(seed)
    x = _cloud(n, d, comps, g)
    y = _dissimilarities(x, sigma, g, ld)
    xe = (x + 0.1 * torch.randn(n, d, generator=g, device=DEV, dtype=torch.float64)).float()
    return xe, y, g


def _pack(y):
    n = y.shape[0]
    iu = torch.triu_indices(n, n, 1, device=DEV)
    return y[iu[0], iu[1]].contiguous()


def _forest(sizes, d, seed):
    """Coalescent trees (two random lineages join after an exponential time;
    every branch at least 0.02 long, as between samples of different dates),
    Sigma, mu; (parent, length, sigma_mat, mu), tips first, in tree order."""
    rng = np.random.default_rng(seed)
    n = sum(sizes)
    parent, length, time, pos = [-1] * n, [0.0] * n, [0.0] * n, 0
    for size in sizes:
        lin = list(range(pos, pos + size))
        pos += size
        t = 0.0
        wait = rng.exponential(size=size)
        pick = rng.random(size=(size, 2))
        for k in range(size, 1, -1):
            t += wait[k - 1] / (k * (k - 1) / 2.0)
            node = len(parent)
            parent.append(-1)
            length.append(0.0)
            time.append(t)
            for h in range(2):
                j = int(pick[k - 1, h] * (k - h))
                lin[j], lin[-1] = lin[-1], lin[j]
                c = lin.pop()
                parent[c] = node
                length[c] = t - time[c] + 0.02
            lin.append(node)
    a = rng.standard_normal((d, d))
    return (np.array(parent, dtype=np.int64), np.array(length), a @ a.T / d + 0.5 * np.eye(d),
            rng.standard_normal(d))


def _tree_locations(n, parent, length, sigma_mat, mu, seed):
    """Brownian diffusion down the trees (parents have larger numbers than children)."""
    rng = np.random.default_rng(seed + 1)
    chol = np.linalg.cholesky(sigma_mat)
    step = rng.standard_normal((len(parent), len(mu))) @ chol.T
    x = np.zeros((len(parent), len(mu)))
    for k in range(len(parent) - 1, -1, -1):
        x[k] = mu + step[k] if parent[k] < 0 else x[parent[k]] + math.sqrt(length[k]) * step[k]
    return x[:n]


TAU0, TAU_U = 1.0, 2.0


def _tree_problem(case, seed):
    sizes = [int(s) for s in case["trees"].split(",")]
    forest = _forest(sizes, case["d"], seed)
    g = _gen(seed)
    x = torch.tensor(_tree_locations(case["n"], *forest, seed), device=DEV)
    y = _dissimilarities(x, case["sigma"], g)
    xe = (x + 0.1 * torch.randn(x.shape, generator=g, device=DEV, dtype=torch.float64)).float()
    return xe, y, g, forest


def _batch_problems(case, seed):
    ns = [int(s) for s in case["ns"].split(",")]
    out = []
    for k, n in enumerate(ns):
        xe, y, g = _problem(n, case["d"], case["comps"], case["sigma"], seed + 7919 * k)
        starts = [(xe + 0.05 * torch.randn(xe.shape, generator=g, device=DEV)).contiguous()
                  for _ in range(case["chains"])]
        out.append((n, y, starts))
    return out


def _held_pairs(case, seed):
    n = case["n"]
    rng = np.random.default_rng(seed)
    m = n * (n - 1) // 2
    i = rng.integers(0, n, size=max(1, int(case["held"] * m)))
    j = rng.integers(0, n - 1, size=i.shape[0])
    j = j + (j >= i)
    return np.stack([i, j], axis=1)


def _draws(case, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((case["iters"], case["n"], case["d"])), rng.uniform(size=case["iters"])


# ----------------------------------------------------------------- the calls


def _model(case, y, xe, prec="fp32c"):
    m = MDS(case["n"], case["d"], prec)
    m.set_data(y, layout="full")
    m.set_sigma(case["sigma"])
    m.set_locations(xe)
    if case.get("order"):
        m.reorder()
    return m


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        probs = _batch_problems(case, seed)
        b = Batch([p[0] for p in probs], case["d"], [case["chains"]] * len(probs))
        for k, (n, y, starts) in enumerate(probs):
            b.set_data(k, y, layout="full")
            b.set_sigma(k, case["sigma"])
        return {"case": case, "batch": b, "starts": [p[2] for p in probs], "seed": seed}
    if kind == "tree":
        xe, y, g, (parent, length, sigma_mat, mu) = _tree_problem(case, seed)
        m = _model(case, y, xe)
        m.set_tree_prior(parent, length, sigma_mat, mu, TAU0, TAU_U)
        p0 = torch.randn(xe.shape, generator=g, device=DEV)
        return {"case": case, "m": m, "x": xe, "p0": p0, "xo": torch.empty_like(xe), "po": torch.empty_like(xe)}
    n, d = case["n"], case["d"]
    xe, y, g = _problem(n, d, case["comps"], case["sigma"], seed, n + case["pad"] if kind == "noalloc" else None)
    st = {"case": case, "x": xe}
    if kind == "noalloc":
        up = y[:, :n].triu(1)
        y[:, :n] = up + up.T
        st.update(x=xe.double(), y=y, g=torch.empty(n, d, device=DEV, dtype=torch.float64))
        return st
    if kind == "load":
        if case["layout"] == "packed":
            y = _pack(y)
        if case["y64"]:
            y = y.double()
        m = MDS(n, d)
        m.set_sigma(case["sigma"])
        st.update(m=m, y=y, g=torch.empty(n, d, device=DEV))
        return st
    prec = case.get("prec", "fp32c")
    if prec == "fp64":
        st["x"] = xe.double()
    st["m"] = _model(case, y, st["x"], prec)
    if kind == "grad":
        st["g"] = torch.empty_like(st["x"])
    elif kind == "autograd":
        st["x"] = xe.requires_grad_()
        st["sigma"] = torch.tensor(case["sigma"], device=DEV, requires_grad=True)
    elif kind == "leapfrog":
        st.update(p0=torch.randn(n, d, generator=g, device=DEV), xo=torch.empty_like(xe), po=torch.empty_like(xe))
    elif kind == "hmc":
        st["p"], st["u"] = _draws(case, seed)
        st["xo"] = torch.empty_like(xe)
    elif kind == "cv":
        st["m"].set_heldout(_held_pairs(case, seed))
        st["g"] = torch.empty_like(xe)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        b = st["batch"]
        for k, starts in enumerate(st["starts"]):
            for c, x in enumerate(starts):
                b.set_locations(k, c, x)
        accepted, _ = b.hmc(1, case["steps"], [case["eps"]] * len(st["starts"]), seed=st["seed"])
        return {"accepted": accepted,
                "x": [[b.get_locations(k, c, dtype=np.float32) for c in range(case["chains"])]
                      for k in range(len(st["starts"]))]}
    if kind == "noalloc":
        ll, ds = ctypes.c_double(), ctypes.c_double()
        x, y, g = st["x"], st["y"], st["g"]
        capi.check(capi.lib().mds_loglik_grad_noalloc(
            case["n"], case["d"], y.data_ptr(), y.shape[1], x.data_ptr(), case["sigma"], g.data_ptr(),
            ctypes.byref(ll), ctypes.byref(ds), torch.cuda.current_stream().cuda_stream))
        return {"loglik": np.float64(ll.value), "grad": g, "dsigma": np.float64(ds.value)}
    m, x = st["m"], st["x"]
    if kind == "autograd":
        loss = mds_loglik(x, st["sigma"], m)
        gx, gs = torch.autograd.grad(loss, (x, st["sigma"]))
        return {"loglik": loss.detach().float(), "grad": gx, "dsigma": gs}
    if kind == "load":
        m.set_data(st["y"], layout=case["layout"])
    m.set_locations(x)
    if kind in ("leapfrog", "tree"):
        m.leapfrog(case["steps"], case["eps"], st["p0"])
        ll, _ = m.log_likelihood()
        return {"x": m.get_locations(out=st["xo"]), "p": m.get_momentum(out=st["po"]), "loglik": ll}
    if kind == "hmc":
        accepted, _, stats = m.hmc(case["iters"], case["steps"], case["eps"], p_all=st["p"], u_all=st["u"])
        return {"accepted": accepted, "x": m.get_locations(out=st["xo"]), "loglik": stats["last_loglik"]}
    ll, g, ds = m.gradient(out=st["g"])
    if kind == "cv":
        m.lpd_reset()
        m.lpd_accumulate()
        lpd, _ = m.lpd()
        return {"loglik": ll, "grad": g, "dsigma": ds, "lpd": lpd}
    if case.get("prec") == "fp64":
        return {"loglik": np.float64(ll), "grad": g, "dsigma": np.float64(ds)}
    return {"loglik": ll, "grad": g, "dsigma": ds}


def work(case):
    """Bytes: Y once per evaluation (4 per pair, or as the caller holds it
    where it is the input), locations in and gradients out.  Operations (an
    FMA as two): per pair and coordinate the difference, its square and the
    two-sided accumulation (7), and about 50 for the root, the residual, Phi,
    log Phi and phi / Phi."""
    kind, d = case["kind"], case["d"]
    if kind == "batch":
        ns = [int(s) for s in case["ns"].split(",")]
        pairs = sum(n * (n - 1) // 2 for n in ns)
        nd = sum(ns) * d * case["chains"]
        return {"bytes": case["steps"] * (4 * pairs + 24 * nd),
                "flops": case["steps"] * case["chains"] * pairs * (7 * d + 50)}
    n = case["n"]
    m = n * (n - 1) // 2
    evals = {"leapfrog": case.get("steps", 0) + 1, "tree": case.get("steps", 0) + 1,
             "hmc": case.get("steps", 0) * case.get("iters", 0) + 1}.get(kind, 1)
    wide = 8 if kind == "noalloc" or case.get("prec") == "fp64" else 4
    b = evals * (4 * m + 4 * wide * n * d)
    if kind == "load":
        b += m * (8 if case["y64"] else 4)
    return {"bytes": b, "flops": evals * m * (7 * d + 50)}


# ------------------------------------------------ 64-bit values, plain torch


def _evaluate(x, y, sigma, keep=None):
    """L, dL/dX, dL/dsigma over pairs i < j (those of `keep` where given), 64 bits."""
    n, d = x.shape
    grad = torch.zeros_like(x)
    sum_r = torch.zeros((), dtype=torch.float64, device=DEV)
    sum_s = torch.zeros((), dtype=torch.float64, device=DEV)
    count = 0
    block = max(64, min(n, (1 << 25) // n))
    for i0 in range(0, n, block):
        i1 = min(n, i0 + block)
        mask = torch.arange(i0, n, device=DEV)[None, :] > torch.arange(i0, i1, device=DEV)[:, None]
        if keep is not None:
            mask &= keep[i0:i1, i0:]
        diff = [x[i0:i1, k, None] - x[None, i0:, k] for k in range(d)]
        d2 = sum(v * v for v in diff)
        dist = d2.sqrt()
        z = dist / sigma
        e = y[i0:i1, i0:n].double() - dist
        log_phi = torch.special.log_ndtr(z)
        ratio = torch.exp(-0.5 * z * z - log_phi) / math.sqrt(2.0 * math.pi)
        zero = torch.zeros((), dtype=torch.float64, device=DEV)
        sum_r += torch.where(mask, e * e / (2.0 * sigma * sigma) + log_phi, zero).sum()
        sum_s += torch.where(mask, e * e / sigma ** 3 + ratio * dist / sigma ** 2, zero).sum()
        w = torch.where(mask & (dist > 0), (ratio / sigma - e / sigma ** 2) / dist, zero)
        count += int(mask.sum())
        for k in range(d):
            t = w * diff[k]
            grad[i0:i1, k] -= t.sum(1)
            grad[i0:, k] += t.sum(0)
    ll = -count * math.log(sigma) - float(sum_r)
    return ll, grad, -count / sigma + float(sum_s)


def _trajectory(x, p, steps, eps, target):
    ll, g = target(x)
    for _ in range(steps):
        p = p + 0.5 * eps * g
        x = x + eps * p
        ll, g = target(x)
        p = p + 0.5 * eps * g
    return x, p, ll


def _philox(q, it, chain, word3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) blocks at counters (q, it, chain, word3); [len(q), 4] uint64."""
    c = [np.asarray(q, dtype=np.uint64)] + [np.full(len(q), v, dtype=np.uint64) for v in (it, chain, word3)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    low = np.uint64(0xFFFFFFFF)
    for _ in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & low, (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return np.stack(c, axis=1)


def _philox_momentum(n, d, chain, seed):
    """Standard normals of iteration 0: element e from counter (e / 4, 0, chain, 0), Box-Muller."""
    w = _philox(np.arange((n * d + 3) // 4), 0, chain, 0, seed)
    u = (w.astype(np.float64) + 0.5) / 2.0 ** 32
    z = np.empty((u.shape[0], 4))
    for h in (0, 2):
        r = np.sqrt(-2.0 * np.log(u[:, h]))
        z[:, h], z[:, h + 1] = r * np.cos(2 * np.pi * u[:, h + 1]), r * np.sin(2 * np.pi * u[:, h + 1])
    return torch.tensor(z.reshape(-1)[:n * d].reshape(n, d), device=DEV)


def exact(case, seed):
    kind = case["kind"]
    sigma = case["sigma"]
    if kind == "batch":
        xs, acc, g = [], [], 0
        for n, y, starts in _batch_problems(case, seed):
            xs.append([])
            for x0 in starts:
                x0 = x0.double()
                p0 = _philox_momentum(n, case["d"], g, seed)
                u = (float(_philox([0], 0, g, 1, seed)[0, 0]) + 0.5) / 2.0 ** 32
                l0 = _evaluate(x0, y, sigma)[0]
                x, p, l1 = _trajectory(x0, p0, case["steps"], case["eps"], lambda v: _evaluate(v, y, sigma)[:2])
                dh = -l1 + l0 + 0.5 * float((p * p).sum()) - 0.5 * float((p0 * p0).sum())
                keep = math.log(u) < -dh
                acc.append(keep)
                xs[-1].append(x if keep else x0)
                g += 1
        return {"accepted": np.array([acc]), "x": xs}
    if kind == "tree":
        xe, y, g, (parent, length, sigma_mat, mu) = _tree_problem(case, seed)
        n, d = xe.shape
        path = torch.zeros(n, len(parent), dtype=torch.float64, device=DEV)
        rows = np.arange(n)
        node = np.arange(n)
        while len(rows):
            path[torch.as_tensor(rows), torch.as_tensor(node)] = 1.0
            node = parent[node]
            rows, node = rows[node >= 0], node[node >= 0]
        root = torch.tensor(parent < 0, device=DEV)
        scale = torch.where(root, torch.tensor(TAU0, dtype=torch.float64, device=DEV), torch.tensor(length, device=DEV))
        lone = torch.tensor(parent[:n] < 0, device=DEV)
        scale[:n] = torch.where(lone, torch.tensor(TAU_U, dtype=torch.float64, device=DEV), scale[:n])
        chol = torch.linalg.cholesky((path * scale) @ path.T)
        s_inv = torch.linalg.inv(torch.tensor(sigma_mat, device=DEV))
        mean = torch.tensor(mu, device=DEV)

        def target(v):
            ll, grad, _ = _evaluate(v, y, sigma)
            return ll, grad - torch.cholesky_solve(v - mean, chol) @ s_inv

        p0 = torch.randn(xe.shape, generator=g, device=DEV).double()
        x, p, ll = _trajectory(xe.double(), p0, case["steps"], case["eps"], target)
        return {"x": x, "p": p, "loglik": ll}
    n, d = case["n"], case["d"]
    xe, y, g = _problem(n, d, case["comps"], sigma, seed)
    x = xe.double()
    if kind == "leapfrog":
        p0 = torch.randn(n, d, generator=g, device=DEV).double()
        x, p, ll = _trajectory(x, p0, case["steps"], case["eps"], lambda v: _evaluate(v, y, sigma)[:2])
        return {"x": x, "p": p, "loglik": ll}
    if kind == "hmc":
        p_all, u_all = _draws(case, seed)
        acc = []
        ll = _evaluate(x, y, sigma)[0]
        for p0, u in zip(p_all, u_all):
            p0 = torch.tensor(p0, device=DEV)
            x1, p1, l1 = _trajectory(x, p0, case["steps"], case["eps"], lambda v: _evaluate(v, y, sigma)[:2])
            dh = -l1 + ll + 0.5 * float((p1 * p1).sum()) - 0.5 * float((p0 * p0).sum())
            acc.append(math.log(u) < -dh)
            if acc[-1]:
                x, ll = x1, l1
        return {"accepted": np.array(acc), "x": x, "loglik": ll}
    keep = None
    if kind == "cv":
        pairs = np.sort(_held_pairs(case, seed), axis=1)
        i, j = (torch.as_tensor(pairs[:, h], device=DEV) for h in (0, 1))
        keep = torch.ones(n, n, dtype=torch.bool, device=DEV)
        keep[i, j] = False
    ll, grad, ds = _evaluate(x, y, sigma, keep)
    out = {"loglik": ll, "grad": grad, "dsigma": ds}
    if kind == "cv":
        i, j = torch.nonzero(~keep, as_tuple=True)
        dist = (x[i] - x[j]).square().sum(1).sqrt()
        lp = (-0.5 * math.log(2 * math.pi) - math.log(sigma) - (y[i, j].double() - dist).square() / (2 * sigma * sigma)
              - torch.special.log_ndtr(dist / sigma))
        out["lpd"] = float(lp.sum())
    if kind == "noalloc" or case.get("prec") == "fp64":
        out["loglik"], out["dsigma"] = np.float64(ll), np.float64(ds)
    return out
