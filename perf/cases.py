"""Timed cases of the CAT library, through its Python entry points.

A program that uses the library does one of four things: it fits a model on calibration rows
(`cat_fit`, or `cat_fit_pca` when the rows are clustered after a PCA), and it corrects rows with a
fitted model (`cat_apply` / `cat_apply_bf16`, or `cat_apply_pca`).  The cases are those calls over
the shapes of the five workloads in `workloads.py` (classifier logits, convolution features, a wide
matrix of several million rows), the PCA of the method's own setting (50 components) and a row
length that is no multiple of four.

Inputs come from the generators of `workloads.py`, on the GPU, from the seed alone.  The model of an
inference case is fitted here with plain torch operations, so it does not depend on the library.
"""
import math

import torch

from paper_2509_26277_b200 import binding as B
from paper_2509_26277_b200 import workloads as W

DEV = "cuda"
MODEL_ROUNDS = 10          # Lloyd rounds behind the model of an inference case


def listed():
    return [
        # Correcting one evaluation batch of logits: launch latency counts.
        dict(name="apply_logits_1k", path="apply", source="head", rows=1024, cols=1000, k=8, din=512, bits=2, alpha=1.0),
        # A validation set (50 000 images) of a 2-bit ResNet-18-like head, with the partial blend
        # that suits 2-bit activations.
        dict(name="apply_logits_50k_blend", path="apply", source="head", rows=50_000, cols=1000, k=16, din=512, bits=2,
             alpha=0.4),
        # The same for a 4-bit ResNet-50-like head: one cloud of points, clusters close together.
        dict(name="apply_logits_50k_w4a4", path="apply", source="head", rows=50_000, cols=1000, k=32, din=2048, bits=4,
             alpha=1.0),
        # Logits with a background class: a row length that is no multiple of four, an odd row count.
        dict(name="apply_ragged_1001", path="apply", source="head", rows=49_999, cols=1001, k=50, din=512, bits=2,
             alpha=1.0),
        # Feature maps of a 3x3x64 convolution (64 images of 56 x 56): short rows, many of them.
        dict(name="apply_conv", path="apply", source="head", rows=200_704, cols=64, k=64, din=576, bits=2, alpha=1.0),
        # The largest: four million rows of 1024, K = 256.
        dict(name="apply_wide_4m", path="apply", source="mixture", rows=4_194_304, cols=1024, k=256, alpha=1.0),
        # Corrected rows handed on in bf16.
        dict(name="apply_wide_bf16", path="apply_bf16", source="mixture", rows=262_144, cols=1024, k=128),
        # Fitting on a small calibration set of logits (1024 samples, 30 rounds).
        dict(name="fit_logits_1k", path="fit", source="head", rows=1024, cols=1000, k=16, din=512, bits=2, iters=30),
        # Fitting on convolution features.
        dict(name="fit_conv", path="fit", source="head", rows=200_704, cols=64, k=64, din=576, bits=2, iters=25),
        # Fitting on a large set, K = 256.
        dict(name="fit_wide_262k", path="fit", source="mixture", rows=262_144, cols=1024, k=256, iters=25),
        # The method as printed: PCA to 50 dimensions, clustering there, the map in the full space.
        dict(name="fit_pca_logits_4k", path="fit_pca", source="head", rows=4096, cols=1000, k=32, din=2048, bits=4,
             iters=30, p=50),
        dict(name="apply_pca_logits_50k", path="apply_pca", source="head", rows=50_000, cols=1000, k=64, din=512, bits=2,
             p=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: K of 1 ... 256, rows of 10 ... 2048 logits, 32 ... 256
    features or 512 ... 1024 wide columns, odd sizes among them."""
    path = rng.choice(["apply", "apply", "apply", "apply_bf16", "fit", "fit", "fit_pca", "apply_pca"])
    c = dict(path=path)
    if path in ("fit_pca", "apply_pca"):
        rows = _log_int(rng, 512, 4096) if path == "fit_pca" else _log_int(rng, 1000, 50_000)
        cols = rng.choice([1000, _log_int(rng, 100, 1000)])
        k = _log_int(rng, 2, 64)
        c.update(source="head", rows=rows, cols=cols, k=k, din=512, bits=rng.choice([2, 4]),
                 p=min(cols, rng.choice([50, _log_int(rng, 8, 64)])))
    else:
        kind = rng.choice(["logits", "logits", "conv", "wide"])
        if kind == "logits":
            rows = _log_int(rng, 512, 100_000)
            cols = rng.choice([1000, 1001, _log_int(rng, 10, 2048)])
            k = _log_int(rng, 1, 256)
            c.update(source="head", rows=rows, cols=cols, k=min(k, rows // 4), din=512, bits=rng.choice([2, 4]))
        elif kind == "conv":
            rows = _log_int(rng, 10_000, 200_000)
            c.update(source="head", rows=rows, cols=rng.choice([32, 48, 64, 96, 128, 256]), k=_log_int(rng, 8, 128),
                     din=576, bits=2)
        else:
            rows = _log_int(rng, 32_768, 262_144 if path == "fit" else 1_000_000)
            c.update(source="mixture", rows=rows, cols=rng.choice([512, 768, 1000, 1024]), k=_log_int(rng, 32, 256))
    if path == "apply":
        c["alpha"] = rng.choice([1.0, 1.0, 0.4])
    if path in ("fit", "fit_pca"):
        c["iters"] = rng.choice([20, 25, 30])
    return c


# ---------------------------------------------------------------- inputs

def _rows(case, seed, fit_rows, apply_rows):
    """(Yq_fit, Yfp_fit, Yq_apply) of the case's generator."""
    s = 7919 * int(seed) + 1
    if case["source"] == "mixture":
        n = max(fit_rows, apply_rows)
        w = W.gaussian_mixture("case", 4, s, n, case["cols"], 256, fit_rows, case["k"], 0, device=DEV)
    else:
        w = W.linear_head("case", 0, s, case["din"], case["cols"], case["bits"], case["bits"], fit_rows, apply_rows,
                          case["k"], 0, device=DEV)
    return w.Yq_fit, w.Yfp_fit, w.Yq_apply


def _lloyd(X, k):
    """Centroids and labels after MODEL_ROUNDS rounds from the first k rows (dense products only:
    the same bits every time)."""
    C = X[:k].clone()
    for t in range(MODEL_ROUNDS + 1):
        lab = torch.argmin((C * C).sum(1) - 2.0 * (X @ C.t()), dim=1)
        one = torch.zeros((X.shape[0], k), dtype=X.dtype, device=X.device)
        one.scatter_(1, lab[:, None], 1.0)
        if t == MODEL_ROUNDS:
            break
        n = one.sum(0)[:, None]
        C = torch.where(n > 0, (one.t() @ X) / n.clamp(min=1.0), C)
    return C.contiguous(), lab, one


def _affine(Yq, Yfp, lab, one):
    n = one.sum(0)[:, None]
    d = n.clamp(min=1.0)
    muq, muf = (one.t() @ Yq) / d, (one.t() @ Yfp) / d
    q, f = Yq - muq[lab], Yfp - muf[lab]
    g = ((one.t() @ (q * f)) / d) / ((one.t() @ (q * q)) / d).clamp(min=1e-8)
    g = torch.where(n > 0, g, torch.ones_like(g))
    b = torch.where(n > 0, muf - g * muq, torch.zeros_like(g))
    return g.contiguous(), b.contiguous()


def prepare(case, seed):
    path, rows, k = case["path"], case["rows"], case["k"]
    st = dict(case=case)
    if path in ("fit", "fit_pca"):
        st["Yq"], st["Yfp"], _ = _rows(case, seed, rows, 1)
        return st
    fit_rows = max(4 * k, min(65_536 if case["source"] == "mixture" else 8192, rows))
    Yq, Yfp, Ya = _rows(case, seed, fit_rows, rows)
    Ya = Ya[:rows]
    if path == "apply_pca":
        mean = Yq.double().mean(0)
        X = Yq.double() - mean
        _, vec = torch.linalg.eigh(X.t() @ X)
        comps = vec[:, -case["p"]:].t().flip(0)
        X = (X @ comps.t()).float()
        st.update(mean=mean.float(), comps=comps.float().contiguous())
    else:
        X = Yq
    C, lab, one = _lloyd(X, k)
    G, Bt = _affine(Yq, Yfp, lab, one)
    out = torch.empty(Ya.shape, dtype=torch.bfloat16 if path == "apply_bf16" else torch.float32, device=DEV)
    st.update(Y=Ya, C=C, G=G, B=Bt, out=out)
    return st


def run(st):
    case = st["case"]
    path = case["path"]
    if path == "apply":
        return B.cat_apply(st["Y"], st["C"], st["G"], st["B"], out=st["out"], want_labels=True, alpha=case["alpha"])
    if path == "apply_bf16":
        return B.cat_apply_bf16(st["Y"], st["C"], st["G"], st["B"], out=st["out"], want_labels=True)
    if path == "apply_pca":
        return B.cat_apply_pca(st["Y"], st["mean"], st["comps"], st["C"], st["G"], st["B"], out=st["out"],
                               want_labels=True)
    if path == "fit_pca":
        return B.cat_fit_pca(st["Yq"], st["Yfp"], case["k"], case["iters"], case["p"])
    return B.cat_fit(st["Yq"], st["Yfp"], case["k"], case["iters"])


def work(case):
    n, d, k = case["rows"], case["cols"], case["k"]
    path = case["path"]
    if path in ("apply", "apply_bf16"):
        return dict(bytes=n * d * (4 + (2 if path == "apply_bf16" else 4)) + 4 * n + 12 * k * d,
                    flops=2.0 * n * d * k + 2.0 * n * d)
    if path == "fit":
        return dict(bytes=8 * n * d + 4 * n + 12 * k * d, flops=2.0 * n * d * k * (case["iters"] + 1) + 6.0 * n * d)
    p = case["p"]
    if path == "apply_pca":
        return dict(bytes=8 * n * d + 4 * n + 8 * k * d + 4 * k * p + 4 * p * d,
                    flops=2.0 * n * d * p + 2.0 * n * p * k + 2.0 * n * d)
    # covariance (one triangle), reduction of a symmetric matrix to tridiagonal form, projection, clustering
    return dict(bytes=8 * n * d + 4 * n + 8 * k * d + 4 * k * p + 4 * p * d,
                flops=1.0 * n * d * d + 4.0 / 3.0 * d ** 3 + 2.0 * n * d * p + 2.0 * n * p * k * (case["iters"] + 1))


def tolerance(case):
    # Labels are decided in fp64, so they are the same whatever the order of the sums; `differ` leaves
    # room for a row on a bisector.  Corrected rows are one fp32 fused multiply-add of those labels'
    # coefficients; the fitted values are fp32 roundings of fp64 sums.
    if case["path"] == "apply_bf16":
        return {"rel": 2e-3, "max": 8e-3, "differ": 1e-5}
    if case["path"] in ("apply", "apply_pca"):
        return {"rel": 1e-6, "max": 1e-5, "differ": 2e-5}
    return {"rel": 1e-5, "max": 1e-4, "differ": 1e-4}


# ---------------------------------------------------------------- the same in fp64

def _nearest64(X, C):
    """Index of the nearest row of C for every row of X (both fp64)."""
    lab = torch.empty(X.shape[0], dtype=torch.int64, device=X.device)
    c2 = (C * C).sum(1)
    for r in range(0, X.shape[0], 65_536):
        lab[r:r + 65_536] = torch.argmin(c2 - 2.0 * (X[r:r + 65_536] @ C.t()), dim=1)
    return lab


def _kmeans64(X, k, iters):
    """Lloyd rounds from the first k rows; the centroids are fp32 between rounds, as the interface
    hands them out."""
    C = X[:k].clone()
    for _ in range(iters):
        one = torch.nn.functional.one_hot(_nearest64(X, C), k).double()
        n = one.sum(0)[:, None]
        C = torch.where(n > 0, (one.t() @ X) / n.clamp(min=1.0), C).float().double()
    return C, _nearest64(X, C)


def _closed_form64(Yq, Yfp, lab, k):
    one = torch.nn.functional.one_hot(lab, k).double()
    n = one.sum(0)[:, None]
    d = n.clamp(min=1.0)
    q, f = Yq.double(), Yfp.double()
    muq, muf = (one.t() @ q) / d, (one.t() @ f) / d
    q, f = q - muq[lab], f - muf[lab]
    g = ((one.t() @ (q * f)) / d) / ((one.t() @ (q * q)) / d).clamp(min=1e-8)
    g = torch.where(n > 0, g, torch.ones_like(g))
    return g, torch.where(n > 0, muf - g * muq, torch.zeros_like(g))


def _pca64(Yq, p):
    mean = Yq.double().mean(0)
    X = Yq.double() - mean
    _, vec = torch.linalg.eigh(X.t() @ X)
    comps = vec[:, -p:].t().flip(0)
    top = torch.gather(comps, 1, comps.abs().argmax(1, keepdim=True))
    return mean, comps * torch.sign(top)


def exact(case, seed):
    """`run`'s outputs in fp64 (what the interface hands on as fp32 in between -- centroids, mean,
    components, projected rows -- is rounded to fp32 there); None for the largest."""
    path, k = case["path"], case["k"]
    if case["rows"] * case["cols"] > 1_100_000_000:
        return None
    st = prepare(case, seed)
    if path in ("fit", "fit_pca"):
        if path == "fit":
            C, lab = _kmeans64(st["Yq"].double(), k, case["iters"])
            g, b = _closed_form64(st["Yq"], st["Yfp"], lab, k)
            return C, g, b, lab.int()
        mean, comps = _pca64(st["Yq"], case["p"])
        Z = ((st["Yq"].double() - mean.float().double()) @ comps.float().double().t()).float()
        C, lab = _kmeans64(Z.double(), k, case["iters"])
        g, b = _closed_form64(st["Yq"], st["Yfp"], lab, k)
        return dict(mean=mean, comps=comps, centroids=C, gamma=g, beta=b, labels=lab.int())
    Y = st["Y"]
    out = torch.empty(Y.shape, dtype=torch.float64, device=DEV)
    lab = torch.empty(Y.shape[0], dtype=torch.int32, device=DEV)
    a = case.get("alpha", 1.0)
    for r in range(0, Y.shape[0], 65_536):
        y = Y[r:r + 65_536].double()
        x = y
        if path == "apply_pca":
            x = ((y - st["mean"].double()) @ st["comps"].double().t()).float().double()
        lb = _nearest64(x, st["C"].double())
        out[r:r + 65_536] = y + a * (st["G"].double()[lb] * y + st["B"].double()[lb] - y)
        lab[r:r + 65_536] = lb.int()
    return out, lab
