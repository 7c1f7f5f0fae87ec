"""The workloads whose time is followed: Kernel K-means through the library's public entry points.

A case is a dict of plain values.  "call" names the entry point ("fit", "batched", "matrix",
"assign", "seeding"); "data" the point cloud:

* "blobs"    isotropic unit-variance Gaussians, centres uniform in [-10, 10]^d;
* "mixture"  centres N(0, 4 I), one sigma in [0.5, 1.5] per component;
* "rings"    concentric rings in the plane (radii 1 .. k, radial noise 0.1), zero-padded to d;
* "images"   integers 0..255 over 255 with 80% zeros, k classes that differ in the pixels they use.

Fits start from an earlier clustering a fifth of which is stale (what a program has that clusters
again after its data moved, or after seeding).  Kernel widths follow the within-cluster distances.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2501_05587_gb300 as pc

# ---- cases ------------------------------------------------------------------------------------


def _fit(data, n, d, k, kernel, passes, **kw):
    c = {"call": "fit", "data": data, "n": n, "d": d, "k": k, "kernel": kernel, "passes": passes,
         "converge": False, "precision": "fp32", "storage": "fp32", "stored": True}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest everyday fit (the paper's 30-pass protocol): latency of a whole call
        dict(_fit("blobs", 2000, 16, 8, "polynomial", 30), name="fit_small"),
        # a few thousand points of ragged size, run until the labels stop changing
        dict(_fit("blobs", 5003, 37, 13, "gaussian", 100, converge=True), name="fit_ragged_converge"),
        # low-dimensional data with a nonlinear structure, K well beyond L2
        dict(_fit("rings", 20000, 8, 4, "gaussian", 30), name="fit_rings"),
        # the headline: an image set of MNIST's shape, FP32 throughout, 50 passes
        dict(_fit("images", 70000, 784, 10, "gaussian", 50), name="fit_images"),
        # the same set with the split-BF16 build and K kept in FP16 (half the bytes a pass)
        dict(_fit("images", 70000, 784, 10, "gaussian", 50, precision="bf16x3", storage="fp16"),
             name="fit_images_half"),
        # many clusters (the paper's k = 100), an odd n
        dict(_fit("blobs", 30011, 64, 100, "polynomial", 30), name="fit_k100"),
        # too many points to store K: tiles recomputed every pass from FP8 rows
        dict(_fit("mixture", 200000, 128, 100, "gaussian", 20, precision="fp8", stored=False),
             name="recompute_fp8"),
        # many independent problems of uneven size in one call (a parameter or subset sweep)
        {"name": "batched_fp32", "call": "batched", "count": 256, "n_lo": 500, "n_hi": 8000, "k_hi": 64,
         "passes": 30, "precision": "fp32", "storage": "fp32"},
        # the same with every K kept in BF16
        {"name": "batched_bf16_k", "call": "batched", "count": 256, "n_lo": 500, "n_hi": 8000, "k_hi": 64,
         "passes": 30, "precision": "fp32", "storage": "bf16"},
        # the kernel matrix alone, for a user's own method on top of it
        {"name": "matrix_fp32", "call": "matrix", "data": "blobs", "n": 20001, "d": 1000, "k": 16,
         "kernel": "linear", "precision": "fp32"},
        # one assignment pass on a user's own (precomputed) kernel matrix, with E
        {"name": "assign_step", "call": "assign", "n": 10007, "d": 32, "k": 32, "kernel": "gaussian",
         "noalloc": False},
        # K-means++ seeding in feature space before a fit
        {"name": "seeding", "call": "seeding", "data": "blobs", "n": 50000, "d": 64, "k": 32,
         "kernel": "gaussian"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["small", "small", "stored", "stored", "half", "clusters", "recompute", "batched",
                       "matrix", "matrix", "assign", "seeding"])
    if call == "small":
        n = _log(rng, 64, 6144)
        return _fit("blobs", n, _log(rng, 16, 128), rng.randint(2, max(2, min(32, n // 32))),
                    rng.choice(["linear", "polynomial", "gaussian"]), rng.choice([30, 100]),
                    converge=rng.random() < 0.5)
    if call in ("stored", "half"):
        n, data = _log(rng, 6200, 50000), rng.choice(["blobs", "images", "rings"])
        half = call == "half"
        return _fit(data, n, 8 if data == "rings" else _log(rng, 256, 900) if data == "images" else _log(rng, 16, 300),
                    4 if data == "rings" else rng.randint(2, 32),
                    "polynomial" if data == "blobs" and not half else "gaussian", rng.choice([20, 30, 50]),
                    precision="fp32" if data == "rings" else rng.choice(["fp32", "fp32", "bf16x3", "bf16"]),
                    storage=rng.choice(["fp16", "bf16"]) if half else "fp32")
    if call == "clusters":
        return _fit("blobs", _log(rng, 9000, 40000), _log(rng, 32, 256), rng.randint(33, 200),
                    rng.choice(["polynomial", "gaussian"]), 30, storage=rng.choice(["fp32", "fp32", "bf16"]))
    if call == "recompute":
        return _fit("mixture", _log(rng, 20000, 160000), _log(rng, 32, 256), rng.randint(8, 128), "gaussian", 20,
                    precision=rng.choice(["fp8", "bf16"]), stored=False)
    if call == "batched":
        lo = _log(rng, 300, 2000)
        return {"call": "batched", "count": _log(rng, 8, 256), "n_lo": lo, "n_hi": _log(rng, 2 * lo, 7000),
                "k_hi": rng.randint(8, 64), "passes": 30, "precision": "fp32", "storage": rng.choice(["fp32", "bf16"])}
    if call == "matrix":
        data = rng.choice(["blobs", "images"])
        return {"call": "matrix", "data": data, "n": _log(rng, 500, 30000),
                "d": _log(rng, 256, 1000) if data == "images" else _log(rng, 8, 2000), "k": 10,
                "kernel": "gaussian" if data == "images" else rng.choice(["linear", "polynomial"]),
                "precision": rng.choice(["fp32", "fp32", "bf16", "bf16x3"])}
    if call == "assign":
        n, noalloc = _log(rng, 500, 20000), rng.random() < 0.3
        return {"call": "assign", "n": n, "d": _log(rng, 16, 64), "k": rng.randint(2, 64 if noalloc else min(200, n // 8)),
                "kernel": rng.choice(["polynomial", "gaussian"]), "noalloc": noalloc}
    return {"call": "seeding", "data": "blobs", "n": _log(rng, 1000, 100000), "d": _log(rng, 16, 256),
            "k": rng.randint(4, 64), "kernel": rng.choice(["polynomial", "gaussian"])}


# ---- inputs -----------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _points(g, data, n, d, k):
    """(n, d) float32 points on the GPU and the component each was drawn from."""
    u = lambda *s: torch.rand(*s, generator=g, device="cuda")  # noqa: E731
    z = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    which = torch.arange(n, device="cuda")[torch.randperm(n, generator=g, device="cuda")] % k
    if data == "rings":
        theta, r = 2 * math.pi * u(n), (which + 1).float() + 0.1 * z(n)
        P = torch.zeros(n, d, device="cuda")
        P[:, 0], P[:, 1] = r * torch.cos(theta), r * torch.sin(theta)
        return P, which
    if data == "images":
        used = u(k, d) < 0.4
        P = torch.floor(256 * u(n, d)) / 255
        return torch.where(used[which] & (u(n, d) < 0.5), P, torch.zeros((), device="cuda")), which
    if data == "mixture":
        C, s = 2 * z(k, d), 0.5 + u(k, 1)
        return C[which] + s[which] * z(n, d), which
    return (20 * u(k, d) - 10)[which] + z(n, d), which


def _stale(g, which, k):
    """The true components with a fifth of the points on a random one, int32."""
    n = which.numel()
    other = torch.randint(0, k, (n,), generator=g, device="cuda")
    stale = torch.rand(n, generator=g, device="cuda") < 0.2
    return torch.where(stale, other, which).to(torch.int32)


def _kernel(kind, data, d):
    if kind == "gaussian":
        sigma = {"rings": 0.5, "images": math.sqrt(d), "mixture": math.sqrt(2 * d), "blobs": math.sqrt(2 * d)}[data]
        return pc.kernel_spec("gaussian", gamma=1.0, sigma=sigma)
    return pc.kernel_spec(kind, gamma=1.0, coef0=1.0, degree=2)


def _instances(case, g):
    """Problems of uneven n, d, k and kernel, as a list of (P, labels, k, kernel).  The sizes
    belong to the case, the points and labels to the seed."""
    sizes = random.Random(case["count"] * 100003 + case["n_lo"] * 1009 + case["n_hi"] + case["k_hi"])
    out = []
    for t in range(case["count"]):
        n, d = sizes.randint(case["n_lo"], case["n_hi"]), sizes.choice([8, 32, 64])
        k = min(sizes.randint(4, case["k_hi"]), n // 32)
        P, which = _points(g, "blobs", n, d, k)
        out.append((P, _stale(g, which, k), k, _kernel("gaussian" if t % 2 else "polynomial", "blobs", d)))
    return out


def prepare(case, seed):
    g = _gen(seed)
    if case["call"] == "batched":
        inst = _instances(case, g)
        labels = torch.empty(sum(P.shape[0] for P, _, _, _ in inst), dtype=torch.int32, device="cuda")
        views = torch.split(labels, [P.shape[0] for P, _, _, _ in inst])
        return {"case": case, "labels": labels,
                "instances": [{"P": P, "init_labels": lab, "k": k, "kernel": kern, "labels_out": v}
                              for (P, lab, k, kern), v in zip(inst, views)]}
    data = case.get("data", "blobs")
    P, which = _points(g, data, case["n"], case["d"], case["k"])
    s = {"case": case, "P": P, "kernel": _kernel(case["kernel"], data, case["d"])}
    if case["call"] in ("fit", "assign"):
        s["labels"] = _stale(g, which, case["k"])
    if case["call"] == "assign":
        n = case["n"]
        s["K"] = torch.empty(n, (n + 3) // 4 * 4, device="cuda")[:, :n]
        for lo in range(0, n, 4096):
            s["K"][lo:lo + 4096] = _kappa(P[lo:lo + 4096].double(), P.double(), s["kernel"])
        s["kdiag"] = s["K"].diagonal().contiguous()
    if case["call"] == "seeding":
        s["u"] = torch.rand(case["k"], generator=g, device="cuda", dtype=torch.float64).cpu().numpy()
    return s


# ---- one pass ---------------------------------------------------------------------------------


def run(s):
    c = s["case"]
    if c["call"] == "fit":
        r = pc.popcorn_fit(s["P"], c["k"], s["kernel"], s["labels"], max_iter=c["passes"], precision=c["precision"],
                           check_convergence=c["converge"], store_k=c["stored"], k_storage=c["storage"])
        return {"labels": r["labels"], "objective": r["objective"], "iterations": r["iterations"]}
    if c["call"] == "batched":
        r = pc.popcorn_fit_batched(s["instances"], max_iter=c["passes"], precision=c["precision"],
                                   check_convergence=False, k_storage=c["storage"])
        return {"labels": s["labels"], "objectives": torch.tensor(r["objectives"]),
                "iterations": torch.tensor(r["iterations"])}
    if c["call"] == "matrix":
        K, kdiag = pc.popcorn_kernel_matrix(s["P"], s["kernel"], precision=c["precision"])
        return {"K": K, "kdiag": kdiag}
    if c["call"] == "assign":
        step = pc.popcorn_assign_step_noalloc if c["noalloc"] else pc.popcorn_assign_step
        r = step(s["K"], s["kdiag"], s["labels"], c["k"], want_E=True)
        return {"labels": r["labels"], "counts": r["counts"], "E": r["E"], "objective": r["J"], "changed": r["changed"]}
    r = pc.popcorn_kmeanspp(s["P"], c["k"], s["kernel"], s["u"])
    return {"labels": r["labels"], "centers": r["centers"]}


# ---- work and exact values --------------------------------------------------------------------


def _fit_work(n, d, passes, elem, stored=True):
    """Points and labels once, and the distinct entries of a stored K once a pass and once more for
    the final objective (once in all when K sits in the 129 MB L2); the products of the build (of
    every pass where K is not stored) and an addition per entry of the square and pass."""
    K = elem * n * (n + 1) // 2
    reads = (passes + 1 if K > 129e6 else 1) if stored else 0
    return {"bytes": 4 * n * d + 8 * n + reads * K,
            "flops": n * (n + 1) * d * (1 if stored else passes + 1) + (passes + 1) * n * n}


def work(case):
    c = case["call"]
    if c == "fit":
        # a fit to convergence from these labels takes three passes
        return _fit_work(case["n"], case["d"], 3 if case["converge"] else case["passes"],
                         4 if case["storage"] == "fp32" else 2, case["stored"])
    if c == "batched":
        lo, hi, e = case["n_lo"], case["n_hi"], 4 if case["storage"] == "fp32" else 2
        n2, n1, p = (lo * lo + lo * hi + hi * hi) / 3, (lo + hi) / 2, case["passes"]   # means over the sizes
        return {"bytes": case["count"] * (e * n2 / 2 * (p + 1) + 4 * 35 * n1 + 8 * n1),
                "flops": case["count"] * (35 * n2 + (p + 1) * n2)}
    n, d, k = case["n"], case["d"], case["k"]
    if c == "matrix":
        return {"bytes": 4 * n * d + 4 * n * n + 4 * n, "flops": n * (n + 1) * d}
    if c == "assign":
        return {"bytes": 4 * n * n + 4 * n * k + 12 * n + 4 * k, "flops": n * n + 3 * n * k}
    return {"bytes": 4 * n * d + 4 * n + 12 * k, "flops": 2 * n * d * k}


def _kappa(X, Y, kern):
    """kappa(X Y^T) in the type of X (float64 here); the Gaussian's distances by norm expansion."""
    B = X @ Y.T
    if kern["kind"] == "linear":
        return B
    if kern["kind"] == "polynomial":
        return B.mul_(kern["gamma"]).add_(kern["coef0"]).pow_(kern["degree"])
    B.mul_(-2).add_((X * X).sum(1)[:, None]).add_((Y * Y).sum(1)[None, :]).clamp_(min=0)
    return B.mul_(-kern["gamma"] / kern["sigma"] ** 2).exp_()


def _matrix64(P, kern):
    X = P.double()
    K = torch.empty(X.shape[0], X.shape[0], dtype=torch.float64, device="cuda")
    for lo in range(0, X.shape[0], 8192):
        K[lo:lo + 8192] = _kappa(X[lo:lo + 8192], X, kern)
    if kern["kind"] == "gaussian":
        K.fill_diagonal_(1.0)
    return K


def _step64(K, diag, labels, k):
    """E = K V^T, D and J of one pass of the method's loop body, in float64."""
    V = torch.nn.functional.one_hot(labels.long(), k).double()
    m = V.sum(0)
    E = (K @ V) / m.clamp(min=1)
    cn = (E * V).sum(0) / m.clamp(min=1)
    D = diag[:, None] - 2 * E + cn[None, :]
    return E, torch.where(m > 0, D, torch.full_like(D, math.inf)), float(D.gather(1, labels.long()[:, None]).sum())


def _fit64(P, kern, labels, k, passes, converge):
    K = _matrix64(P, kern)
    diag = K.diagonal().clone()
    done = 0
    while done < passes:
        _, D, J = _step64(K, diag, labels, k)
        new = D.argmin(1).to(torch.int32)
        done += 1
        if torch.equal(new, labels):
            return new, J, done if converge else passes
        labels = new
    return labels, _step64(K, diag, labels, k)[2], done


def exact(case, seed):
    if case["call"] == "seeding" or (case["call"] == "fit" and case["n"] > (75000 if case["stored"] else 60000)):
        return None
    s = prepare(case, seed)
    if case["call"] == "fit":
        labels, J, its = _fit64(s["P"], s["kernel"], s["labels"], case["k"], case["passes"], case["converge"])
        return {"labels": labels, "objective": J, "iterations": its}
    if case["call"] == "batched":
        got = [_fit64(x["P"], x["kernel"], x["init_labels"], x["k"], case["passes"], False) for x in s["instances"]]
        return {"labels": torch.cat([r[0] for r in got]), "objectives": torch.tensor([r[1] for r in got]).double(),
                "iterations": torch.tensor([r[2] for r in got])}
    if case["call"] == "matrix":
        K = _matrix64(s["P"], s["kernel"])
        return {"K": K, "kdiag": K.diagonal().contiguous()}
    E, D, J = _step64(s["K"].double(), s["kdiag"].double(), s["labels"], case["k"])
    new = D.argmin(1).to(torch.int32)
    return {"labels": new, "counts": torch.bincount(new.long(), minlength=case["k"]).to(torch.int32), "E": E,
            "objective": J, "changed": int((new != s["labels"]).sum())}
