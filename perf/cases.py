"""The calls whose time counts: what a program that clusters with this
package asks of it, over the range of sizes it is used at.

Each case is a dict of plain values.  ``prepare`` makes what the program holds
before the call (points on the GPU or in host memory, a context, a network),
``run`` makes the call through the package's public entry points and returns
its outputs whole, ``work`` states the bytes and operations the call cannot
do without, and ``exact`` gives the same outputs from plain float64 torch.

Kinds of case
  run       km_run from given starting centres: Lloyd's loop to its stop test
            or its step limit (the fused path for d <= 4 and K <= 256, the
            tensor-core path for d = 64, the general path elsewhere)
  steps     a loop the program drives itself, one km_step per iteration
  batch     many unequal instances in one KMeansBatch run
  seed      k-means++ seeding of resident points
  grad      loss and gradients of the set network on a batch of samples
  predict   starting centres from the set network for a batch of samples
  fit       one whole fit from host arrays: context, points in, k-means++,
            Lloyd's loop, labels out, objective
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2405_12052_gb300 as km
from paper_2405_12052_gb300 import learned

DEV = "cuda"

# ---------------------------------------------------------------- the cases


def listed():
    return [
        # The paper's smallest set (2-D, 1e5 points, 8 Gaussians): a run of
        # about twenty steps of a few microseconds each, labels to the host.
        {"name": "run_2d_n1e5_k8", "kind": "run", "n": 100_000, "d": 2, "k": 8, "mix": "iso", "box": 10.0,
         "max_iter": 100, "tol": 1e-6, "steps": 20, "labels": "host", "label_bytes": 4},
        # The paper's largest set (3-D, 1e6 points) with its largest cluster
        # count; one point more than a round number.
        {"name": "run_3d_n1e6_k11", "kind": "run", "n": 1_000_001, "d": 3, "k": 11, "mix": "aniso", "box": 10.0,
         "max_iter": 100, "tol": 1e-6, "steps": 100, "labels": "host", "label_bytes": 4},
        # Big data: 1e8 points in 3-D, K = 32 from a k-means++ start, to its
        # own convergence or the configuration's limit of 300 steps; byte labels stay on the GPU.
        {"name": "run_3d_n1e8_k32", "kind": "run", "n": 100_000_000, "d": 3, "k": 32, "mix": "aniso", "box": 50.0,
         "max_iter": 300, "tol": 1e-6, "steps": 100, "labels": "device", "label_bytes": 1},
        # Cancellation stress: 2^27 points around 1e4 with K = 256, in a loop
        # that looks at the error after every step.
        {"name": "steps_offset_3d_n2p27_k256", "kind": "steps", "n": 1 << 27, "d": 3, "k": 256, "mix": "iso",
         "box": 50.0, "offset": 1e4, "steps": 3, "labels": "device", "label_bytes": 1},
        # Embeddings: 1e7 vectors of 64 dimensions into 1024 clusters on the
        # tensor cores.
        {"name": "run_64d_n1e7_k1024", "kind": "run", "n": 10_000_000, "d": 64, "k": 1024, "mix": "iso", "box": 10.0,
         "max_iter": 8, "tol": 1e-6, "steps": 8, "labels": "device", "label_bytes": 4},
        # A codebook over a smaller set of 64-dimensional vectors, FP16
        # operands, ragged in N and K.
        {"name": "run_64d_n200003_k100", "kind": "run", "n": 200_003, "d": 64, "k": 100, "mix": "iso", "box": 8.0,
         "max_iter": 20, "tol": 1e-6, "steps": 20, "labels": "device", "label_bytes": 4, "tc_operands": "f16"},
        # Feature vectors of a dimension without a kernel of its own.
        {"name": "run_16d_n1000003_k64", "kind": "run", "n": 1_000_003, "d": 16, "k": 64, "mix": "iso", "box": 5.0,
         "sigma": 1.5, "max_iter": 10, "tol": 1e-6, "steps": 10, "labels": "device", "label_bytes": 4},
        # 256 unequal instances (1e3 to 1e6 points, K 4 to 64), each to its
        # own convergence.
        {"name": "batch_256", "kind": "batch", "count": 256, "n_lo": 1_000, "n_hi": 1_000_000, "k_lo": 4, "k_hi": 64,
         "size_seed": 0, "max_iter": 300, "tol": 1e-6, "steps": 50},
        # The k-means++ start of the 1e8-point run.
        {"name": "seed_3d_n1e8_k32", "kind": "seed", "n": 100_000_000, "d": 3, "k": 32, "mix": "aniso", "box": 50.0},
        # One training batch of the learned initialiser, as its committed
        # weights were made (256 samples of 4096 points).
        {"name": "grad_256x4096", "kind": "grad", "sets": 256, "points": 4096, "d": 3, "k": 16},
        # The learned start's forward pass on 64 rotated copies of a sample.
        {"name": "predict_64x4096", "kind": "predict", "sets": 64, "points": 4096, "d": 3, "k": 16},
        # One fit from numpy arrays of rows, as a script would call it once.
        {"name": "fit_host_3d_n1e6_k16", "kind": "fit", "n": 1_000_000, "d": 3, "k": 16, "mix": "aniso", "box": 50.0,
         "max_iter": 50, "tol": 1e-6, "steps": 20},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run64", "run64", "rungen", "steps", "batch", "seed", "grad", "predict", "fit"])
    if kind == "run":
        n, d, k = _logint(rng, 10_000, 50_000_000), rng.randint(1, 4), _logint(rng, 2, 256)
        # at most the work of the largest listed run
        steps = max(5, min(100, int(4e11 / (n * k))))
        return {"kind": "run", "n": n, "d": d, "k": k, "mix": rng.choice(["iso", "aniso"]),
                "box": rng.choice([10.0, 50.0]), "max_iter": steps, "tol": 1e-6, "steps": steps,
                "labels": "host" if n <= 1_000_000 else "device", "label_bytes": rng.choice([4, 1])}
    if kind == "run64":
        n, k = _logint(rng, 20_000, 10_000_000), _logint(rng, 16, 1024)
        return {"kind": "run", "n": n, "d": 64, "k": k, "mix": "iso", "box": rng.choice([8.0, 10.0]), "max_iter": 8,
                "tol": 1e-6, "steps": 8, "labels": "device", "label_bytes": 4,
                "tc_operands": rng.choice(["bf16", "f16"])}
    if kind == "rungen":
        n, d, k = _logint(rng, 10_000, 2_000_000), rng.randint(5, 48), _logint(rng, 3, 300)
        return {"kind": "run", "n": n, "d": d, "k": k, "mix": "iso", "box": 5.0, "sigma": 1.5, "max_iter": 5,
                "tol": 1e-6, "steps": 5, "labels": "device", "label_bytes": 4}
    if kind == "steps":
        n, k = _logint(rng, 50_000, 1 << 27), _logint(rng, 8, 256)
        return {"kind": "steps", "n": n, "d": rng.randint(2, 3), "k": k, "mix": "iso", "box": 50.0,
                "offset": rng.choice([0.0, 1e4]), "steps": 3, "labels": "device", "label_bytes": 1}
    if kind == "batch":
        n_hi = rng.choice([4_000, 30_000, 300_000])
        return {"kind": "batch", "count": _logint(rng, 16, 256), "n_lo": 1_000, "n_hi": n_hi, "k_lo": 4,
                "k_hi": rng.choice([16, 64]), "size_seed": rng.randint(1, 1000), "max_iter": 100, "tol": 1e-6,
                "steps": 50}
    if kind == "seed":
        return {"kind": "seed", "n": _logint(rng, 100_000, 100_000_000), "d": rng.randint(2, 3),
                "k": _logint(rng, 4, 32), "mix": "aniso", "box": 50.0}
    if kind in ("grad", "predict"):
        return {"kind": kind, "sets": _logint(rng, 1 if kind == "predict" else 8, 256),
                "points": 64 * rng.randint(8, 64), "d": 3, "k": 16}
    n = _logint(rng, 10_000, 3_000_000)
    return {"kind": "fit", "n": n, "d": rng.randint(2, 3), "k": _logint(rng, 4, 32), "mix": "aniso", "box": 50.0,
            "max_iter": 50, "tol": 1e-6, "steps": 20}


# ------------------------------------------------------------------- inputs


def _points(case, g, n=None, d=None, comps=None):
    """(d, n) float32 points of a Gaussian mixture with as many components as
    clusters: isotropic (unit or given sigma, equal weights) or anisotropic
    (random axes, sigmas in [0.5, 2], Dirichlet(1) weights)."""
    n, d = n or case["n"], d or case["d"]
    c = comps or case["k"]
    mu = (torch.rand(c, d, generator=g, device=DEV) * 2 - 1) * case.get("box", 10.0)
    x = torch.empty(d, n, device=DEV)
    aniso = case.get("mix") == "aniso"
    if aniso:
        w = -torch.log(torch.rand(c, generator=g, device=DEV, dtype=torch.float64).clamp_(1e-12))
        cdf = torch.cumsum(w / w.sum(), 0).float()
        axes = torch.linalg.qr(torch.randn(c, d, d, generator=g, device=DEV).cpu())[0].to(DEV)
        axes = axes * (torch.rand(c, 1, d, generator=g, device=DEV) * 1.5 + 0.5)
    off = case.get("offset", 0.0)
    for a in range(0, n, 1 << 23):
        m = min(1 << 23, n - a)
        u = torch.rand(m, generator=g, device=DEV)
        z = torch.randn(d, m, generator=g, device=DEV)
        if aniso:
            comp = torch.searchsorted(cdf, u).clamp_(max=c - 1)
            for j in range(d):
                y = mu[:, j][comp]
                for i in range(d):
                    y = y + axes[:, j, i][comp] * z[i]
                x[j, a:a + m] = y + off
        else:
            comp = (u * c).long().clamp_(max=c - 1)
            for j in range(d):
                x[j, a:a + m] = mu[:, j][comp] + case.get("sigma", 1.0) * z[j] + off
    return x


def _distinct(x, k, g):
    """K distinct points as the start (K x d float64, on the host)."""
    idx = torch.randperm(x.shape[1], generator=g, device=DEV)[:k]
    return x[:, idx].t().double().cpu().numpy()


def _spread(x, k, g):
    """A k-means++ start drawn from a subsample (K x d float64, host)."""
    s = x[:, torch.randint(x.shape[1], (min(x.shape[1], 1 << 17),), generator=g, device=DEV)].double()
    u = torch.rand(k, generator=g, device=DEV, dtype=torch.float64)
    pick = (u[0] * s.shape[1]).long()
    d2 = None
    out = []
    for c in range(k):
        m = s[:, pick]
        out.append(m)
        t = ((s - m[:, None]) ** 2).sum(0)
        d2 = t if d2 is None else torch.minimum(d2, t)
        cum = torch.cumsum(d2, 0)
        if c + 1 < k:
            pick = torch.searchsorted(cum, u[c + 1] * cum[-1]).clamp_(max=s.shape[1] - 1)
    return torch.stack(out).cpu().numpy()


def _sizes(case):
    r = np.random.default_rng(case["size_seed"])
    n = np.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["count"])).astype(np.int64)
    d = r.integers(2, 4, case["count"]).astype(np.int64)
    k = np.minimum(r.integers(case["k_lo"], case["k_hi"] + 1, case["count"]), n)
    return n, d, k


def _inputs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    kind = case["kind"]
    if kind in ("run", "steps"):
        x = _points(case, g)
        start = _spread if case["d"] <= 4 and case["k"] >= 32 else _distinct
        return {"x": x, "mu0": start(x, case["k"], g)}
    if kind in ("seed", "fit"):
        x = _points(case, g)
        u = np.random.default_rng(seed).random(case["k"])
        return {"x": x, "u": u}
    if kind == "batch":
        n, d, k = _sizes(case)
        xs = [_points({"box": 10.0}, g, int(n[i]), int(d[i]), int(k[i])) for i in range(len(n))]
        return {"x": torch.cat([x.reshape(-1) for x in xs]), "mu0": [_distinct(x, int(k[i]), g)
                                                                    for i, x in enumerate(xs)]}
    x, means = learned.mixtures(case["sets"], S=case["points"], d=case["d"], k=case["k"], seed=seed, device=DEV)
    return {"x": x, "t": means.float()}


def prepare(case, seed):
    st = {"case": case, **_inputs(case, seed)}
    kind = case["kind"]
    if kind in ("run", "steps", "seed"):
        g = km.KMeans(case["n"], case["d"], case["k"], label_bytes=case.get("label_bytes", 4),
                      tc_operands=case.get("tc_operands", "bf16"))
        g.set_points(st["x"], borrow=True)
        st["g"] = g
        if case.get("labels") == "device":
            st["labels"] = torch.empty(case["n"], device=DEV,
                                       dtype=torch.uint8 if case["label_bytes"] == 1 else torch.int32)
    elif kind == "fit":
        st["x"] = np.ascontiguousarray(st["x"].t().cpu().numpy())
    elif kind == "batch":
        n, d, k = _sizes(case)
        b = km.KMeansBatch(n, d, k)
        b.set_points(st["x"])
        b.set_init(st["mu0"])
        b.tune()
        st["b"] = b
    else:
        net = learned.load()  # the committed weights (d = 3, K = 16)
        st["net"] = net
    torch.cuda.synchronize()
    return st


# ----------------------------------------------------------------- the call


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "run":
        g = st["g"]
        g.set_init(st["mu0"])
        host = case["labels"] == "host"
        r = g.run(case["max_iter"], case["tol"], want_labels=host)
        if host:
            z = r["labels"]
        else:
            z = st["labels"]
            g.labels_into(z)
        return [z, r["centroids"], r["iters"], r["E"]]
    if kind == "steps":
        g = st["g"]
        g.set_init(st["mu0"])
        errs = [g.step() for _ in range(case["steps"])]
        g.labels_into(st["labels"])
        return [st["labels"], g.centroids(), g.counts(), [e for e, _ in errs], [e2 for _, e2 in errs]]
    if kind == "batch":
        b = st["b"]
        b.set_init(st["mu0"])
        r = b.run(case["max_iter"], case["tol"])
        return [r["labels"], r["centroids"], r["iters"], r["E"]]
    if kind == "seed":
        mu, idx = st["g"].init_kmeanspp(st["u"])
        return [mu, idx]
    if kind == "grad":
        loss = st["net"].loss_grad(st["x"], st["t"])
        return [loss, st["net"].grads()]
    if kind == "predict":
        return [st["net"].predict(st["x"])]
    g = km.KMeans(case["n"], case["d"], case["k"])
    g.set_points(st["x"], layout="nxd")
    mu0, idx = g.init_kmeanspp(st["u"])
    r = g.run(case["max_iter"], case["tol"])
    obj = g.objective()
    g.close()
    return [idx, r["labels"], r["centroids"], r["iters"], r["E"], obj]


# --------------------------------------------------------------- the bounds


def work(case):
    """Bytes: the points read once, labels and centroids written once.
    Operations: a subtraction, a product and a sum per point, centroid and
    coordinate and step (``steps`` is the number a run of these inputs takes
    where it ends by its own test), or two per weight of a matrix product."""
    kind = case["kind"]
    if kind in ("run", "steps", "fit"):
        n, d, k = case["n"], case["d"], case["k"]
        per = 2 if d == 64 else 3
        flops = per * n * k * d * case["steps"]
        if kind == "fit":
            flops += 3 * n * (k - 1) * d
        return {"bytes": 4 * n * d + n * case.get("label_bytes", 4) + 16 * k * d, "flops": flops}
    if kind == "batch":
        n, d, k = _sizes(case)
        return {"bytes": int((4 * n * d + 4 * n).sum()), "flops": int((3 * n * d * k).sum()) * case["steps"]}
    if kind == "seed":
        n, d, k = case["n"], case["d"], case["k"]
        return {"bytes": 4 * n * d, "flops": 3 * n * d * (k - 1)}
    p, d, k, b, h = case["sets"] * case["points"], case["d"], case["k"], case["sets"], 128
    fwd = 2 * p * (d * h + h * h) + 2 * b * (h * h + h * k * d)
    params = 2 * h * h + 3 * h + h * d + k * d * h + k * d
    if kind == "predict":
        return {"bytes": 4 * p * d + 4 * params + 8 * b * k * d, "flops": fwd}
    # the gradient to the points is not needed: one product less than twice
    return {"bytes": 4 * p * d + 4 * b * k * d + 8 * params,
            "flops": 3 * fwd - 2 * p * d * h}


# ------------------------------------------------------- the float64 answers


def _assign64(x, mu):
    """Nearest centre per point: sum_j (x_j - m_j)^2 in float64, in order."""
    n, k = x.shape[1], mu.shape[0]
    step = max(1, (1 << 26) // k)
    out = torch.empty(n, dtype=torch.int64, device=DEV)
    for a in range(0, n, step):
        xs = x[:, a:a + step].double()
        acc = None
        for j in range(x.shape[0]):
            t = xs[j][:, None] - mu[:, j][None, :]
            t = t * t
            acc = t if acc is None else acc + t
        out[a:a + step] = acc.argmin(1)
    return out


def _lloyd64(x, mu0, max_iter, tol):
    mu = torch.as_tensor(mu0, dtype=torch.float64, device=DEV)
    k = mu.shape[0]
    errs = []
    for _ in range(max_iter):
        z = _assign64(x, mu)
        cnt = torch.bincount(z, minlength=k)
        s = torch.stack([torch.bincount(z, weights=x[j].double(), minlength=k) for j in range(x.shape[0])], 1)
        new = torch.where(cnt[:, None] > 0, s / cnt[:, None].clamp(min=1), mu)
        e2 = float(((new - mu) ** 2).sum())
        errs.append((math.sqrt(e2), e2))
        mu = new
        if errs[-1][0] < tol:
            break
    return z, mu, cnt, errs


def _net64(prm, x, d, k, t=None):
    h = 128
    p = torch.as_tensor(prm, dtype=torch.float64, device=DEV).requires_grad_(t is not None)
    at, w = 0, []
    for shape in ((h, d), (h,), (h, h), (h,), (h, h), (h,), (k * d, h), (k * d,)):
        size = math.prod(shape)
        w.append(p[at:at + size].reshape(shape))
        at += size
    mean = x.double().mean(1, keepdim=True)
    sd = x.double().std(1, unbiased=False, keepdim=True)
    sd = torch.where(sd > 0, sd, torch.ones_like(sd))
    loss, outs = 0.0, []
    for a in range(0, x.shape[0], 32):
        xs = (x[a:a + 32].double() - mean[a:a + 32]) / sd[a:a + 32]
        h2 = torch.relu(torch.relu(xs @ w[0].T + w[1]) @ w[2].T + w[3])
        o = torch.relu(h2.mean(1) @ w[4].T + w[5]) @ w[6].T + w[7]
        o = o.reshape(-1, k, d)
        if t is None:
            outs.append((o * sd[a:a + 32] + mean[a:a + 32]).detach())
            continue
        ts = (t[a:a + 32].double() - mean[a:a + 32]) / sd[a:a + 32]
        dist = ((o[:, :, None, :] - ts[:, None, :, :]) ** 2).sum(-1)
        part = (dist.amin(2).sum() + dist.amin(1).sum()) / k / x.shape[0]
        part.backward(retain_graph=True)
        loss += float(part.detach())
    return torch.cat(outs) if t is None else (loss, p.grad)


def _seed64(x, u, k):
    n = x.shape[1]
    i = min(int(math.floor(u[0] * n)), n - 1)
    idx, d2 = [i], None
    for c in range(1, k):
        m = x[:, i].double()
        acc = None
        for j in range(x.shape[0]):
            t = x[j].double() - m[j]
            t = t * t
            acc = t if acc is None else acc + t
        d2 = acc if d2 is None else torch.minimum(d2, acc)
        cum = torch.cumsum(d2, 0)
        i = min(int(torch.searchsorted(cum, float(u[c]) * cum[-1], right=True)), n - 1)
        idx.append(i)
    idx = torch.tensor(idx, device=DEV)
    return x[:, idx].t().double().cpu().numpy(), idx.cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("run", "steps") and 3 * case["n"] * case["k"] * case["d"] * case["steps"] > 1.2e12:
        return None
    inp = _inputs(case, seed)
    x = inp["x"]
    # labels, picks and counts are whole numbers: they stay what they are
    if kind == "run":
        _, mu, _, errs = _lloyd64(x, inp["mu0"], case["max_iter"], case["tol"])
        return [None, mu.cpu().numpy(), None, errs[-1][0]]
    if kind == "steps":
        _, mu, _, errs = _lloyd64(x, inp["mu0"], case["steps"], -1.0)
        return [None, mu.cpu().numpy(), None, [e for e, _ in errs], [e2 for _, e2 in errs]]
    if kind == "batch":
        n, d, k = _sizes(case)
        at, mus, es = 0, [], []
        for i in range(len(n)):
            xi = x[at:at + int(n[i] * d[i])].reshape(int(d[i]), int(n[i]))
            at += int(n[i] * d[i])
            _, mu, _, errs = _lloyd64(xi, inp["mu0"][i], case["max_iter"], case["tol"])
            mus.append(mu.cpu().numpy().reshape(-1))
            es.append(errs[-1][0])
        return [None, np.concatenate(mus), None, np.array(es)]
    if kind == "seed":
        mu, _ = _seed64(x, inp["u"], case["k"])
        return [mu, None]
    if kind in ("grad", "predict"):
        prm = np.load(learned.WEIGHTS)["params"]
        if kind == "predict":
            return [_net64(prm, x, case["d"], case["k"]).cpu().numpy()]
        loss, grad = _net64(prm, x, case["d"], case["k"], inp["t"])
        return [loss, grad.cpu().numpy()]
    mu0, _ = _seed64(x, inp["u"], case["k"])
    z, mu, _, errs = _lloyd64(x, mu0, case["max_iter"], case["tol"])
    obj = float(((x.double() - mu[z].t()) ** 2).sum())
    return [None, None, mu.cpu().numpy(), None, errs[-1][0], obj]
