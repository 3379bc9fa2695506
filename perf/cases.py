"""The calls whose time matters to a user of this library, as measurable cases.

Every case is a dict of plain values with a ``kind``:

* ``run``       -- Algorithm 1 from a given start: set_basis, T iterations,
                   the history, the pairs and the final basis (Sec. IV, V);
* ``step``      -- one synchronous iteration from a given basis, the call of
                   a user who drives the loop from outside;
* ``batch``     -- many uneven noisy scenes run together (Sec. VII);
* ``sweep``     -- dimension estimation over k = 1..kmax on one point set
                   (Sec. VI-A, VI-B);
* ``subsets``   -- the same on repeated random subsets of pixels (Sec. VI-C);
* ``softmin``   -- value and gradient of the soft-min objective through
                   torch.autograd;
* ``ascent``    -- Riemannian ascent steps on that objective;
* ``pca``       -- the secant-PCA start (Algorithm 1's initialisation);
* ``threshold`` -- the noisy-data variant at a new length threshold: lengths
                   prepared again, then the worst secant of the basis.

Data are the synthetic families of ``workloads.py`` (trigonometric moment
curve, blob images, hyperspectral mixtures), drawn here on the GPU from the
seed.  ``exact`` restates each computation in 64 bits with plain torch/numpy.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1807_03425_gb300 import BF16, Sap, SapBatch
from paper_1807_03425_gb300.autograd import softmin

DEV = "cuda"


# ------------------------------------------------------------------ cases --

def listed():
    return [
        # the paper's kind of small FP64 experiment: 200 points of a curve,
        # a full loop of a hundred iterations (launches and latency count)
        dict(name="small_f64_loop", kind="run", data="curve", N=200, n=10, k=3, dtype="f64", path="plain",
             mode="literal", split="fp16", eps=0.0, noise=0.0, alpha=0.01, T=100),
        # one synchronous iteration on a small FP32 set: the smallest call
        dict(name="small_step", kind="step", data="curve", N=700, n=20, k=4, dtype="f32", path="restructured",
             mode="literal", split="fp16", eps=0.0, noise=0.0, alpha=0.005, T=1),
        # the main workload: SAP on 8192 points of a curve in R^100
        dict(name="curve_loop", kind="run", data="curve", N=8192, n=100, k=5, dtype="f32", path="restructured",
             mode="literal", split="fp16", eps=0.0, noise=0.0, alpha=0.005, T=32),
        # the form that stores nothing per pair (no room for N^2/2 lengths),
        # on an odd number of points
        dict(name="plain_loop", kind="run", data="curve", N=4001, n=100, k=5, dtype="f32", path="plain",
             mode="literal", split="fp16", eps=0.0, noise=0.0, alpha=0.005, T=4),
        # the largest single scene: 16-bit pixels, wide basis, short secants
        # discarded, the other reading of the rotation
        dict(name="scene_loop", kind="run", data="scene", N=19939, n=224, k=10, dtype="bf16", path="restructured",
             mode="angle", split="fp16", eps=0.05, noise=0.01, alpha=0.01, T=8),
        # many uneven scenes run together
        dict(name="scene_batch", kind="batch", B=16, N_min=500, N_max=12000, n=224, k=10, eps=0.05, alpha=0.01, T=8),
        # dimension estimation on images: 20 bases over 4096 points in R^4096
        dict(name="image_sweep", kind="sweep", data="images", N=4096, side=64, kmax=20, alpha=0.01, threshold=0.1,
             T=8),
        # dimension estimation repeated on random subsets of the pixels
        dict(name="subset_sweep", kind="subsets", N=21025, n=200, R=3, m=512, kmax=10, alpha=0.01, threshold=0.1,
             T=24),
        # gradient of the smooth objective, as a training loop asks for it
        dict(name="softmin_grad", kind="softmin", data="curve", N=16384, n=100, k=5, dtype="f32", noise=0.0,
             tau=0.01),
        # ascent on 16-bit pixels at a ragged size and the widest basis
        dict(name="softmin_ascent", kind="ascent", data="scene", N=5001, n=150, k=8, dtype="bf16", noise=0.01,
             tau=0.02, eta=0.005, T=10),
        # the starting basis of Algorithm 1
        dict(name="pca_start", kind="pca", data="curve", N=8192, n=100, k=5, dtype="f32", noise=0.0),
        # a noisy set judged at a new threshold
        dict(name="threshold_change", kind="threshold", data="curve", N=8000, n=90, k=6, dtype="f32", noise=0.05,
             eps=0.8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "step", "batch", "sweep", "subsets", "softmin", "ascent", "pca",
                       "threshold"])
    data = rng.choice(["curve", "scene"])
    noise = 0.01 if data == "scene" else rng.choice([0.0, 0.02])
    if kind in ("run", "step"):
        path = rng.choice(["restructured", "restructured", "restructured", "plain"])
        dtype = rng.choice(["f32", "f32", "bf16"]) if path == "restructured" else rng.choice(["f32", "f64"])
        N = _log_int(rng, 150, 12000 if path == "restructured" else 4000 if dtype == "f32" else 800)
        n = _log_int(rng, 8, 400 if dtype != "f64" else 48)
        k = min(n // 2, rng.randint(2, 8) if path == "plain" or rng.random() < 0.6 else rng.randint(9, 32))
        # the 16-bit split of less precision marks most pairs as near: its
        # list has room for all pairs of 5000 points
        split = rng.choice(["fp16", "fp16", "bf16"]) if N <= 5000 else "fp16"
        return dict(kind=kind, data=data, N=N, n=n, k=k, dtype=dtype, path=path,
                    mode=rng.choice(["literal", "literal", "angle"]), split=split,
                    eps=rng.choice([0.0, 0.05]), noise=noise, alpha=rng.choice([0.005, 0.01]),
                    T=1 if kind == "step" else rng.choice([2, 3, 4, 16, 40]))
    if kind == "batch":
        return dict(kind=kind, B=rng.randint(2, 10), N_min=_log_int(rng, 150, 600), N_max=_log_int(rng, 900, 6000),
                    n=_log_int(rng, 24, 256), k=rng.randint(2, 12), eps=0.05, alpha=0.01,
                    T=rng.choice([2, 3, 4, 16]))
    if kind == "sweep":
        return dict(kind=kind, data="images", N=_log_int(rng, 200, 2500), side=rng.randint(12, 64),
                    kmax=rng.randint(3, 20), alpha=0.01, threshold=0.1, T=rng.randint(2, 6))
    if kind == "subsets":
        return dict(kind=kind, N=_log_int(rng, 2000, 21025), n=_log_int(rng, 30, 224), R=rng.randint(1, 3),
                    m=_log_int(rng, 200, 1000), kmax=rng.randint(3, 12), alpha=0.01, threshold=0.1,
                    T=rng.choice([2, 3, 4, 16]))
    if kind in ("softmin", "ascent"):
        c = dict(kind=kind, data=data, N=_log_int(rng, 300, 12000), n=_log_int(rng, 6, 300), dtype=rng.choice(["f32", "bf16"]),
                 noise=0.01 if data == "scene" else rng.choice([0.0, 0.02]), tau=rng.choice([0.01, 0.02, 0.05]))
        c["k"] = min(c["n"] // 2, rng.randint(1, 8))
        if kind == "ascent":
            c.update(N=min(c["N"], 6000), eta=0.005, T=rng.randint(2, 8))
        return c
    if kind == "pca":
        n = _log_int(rng, 6, 160)
        return dict(kind=kind, data=data, N=_log_int(rng, 200, 5000), n=n, k=min(n // 2, rng.randint(1, 8)),
                    dtype=rng.choice(["f32", "f64"]), noise=0.01 if data == "scene" else 0.0)
    n = _log_int(rng, 12, 300)
    return dict(kind=kind, data="curve", N=_log_int(rng, 300, 8000), n=n, k=min(n // 2, rng.randint(2, 12)),
                dtype=rng.choice(["f32", "bf16"]), noise=0.05, eps=rng.choice([0.2, 0.5]))


# ----------------------------------------------------------------- inputs --

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _store(X, dtype):
    return X.to({"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[dtype]).contiguous()


def _curve(N, n, noise, g):
    t = torch.rand(N, 1, generator=g, device=DEV, dtype=torch.float64) * (2 * math.pi)
    q = torch.arange(1, (n + 1) // 2 + 1, device=DEV, dtype=torch.float64)
    X = torch.stack([torch.cos(t * q), torch.sin(t * q)], dim=2).reshape(N, -1)[:, :n]
    if noise > 0:
        X = X + noise * torch.randn(N, n, generator=g, device=DEV, dtype=torch.float64)
    return X


def _endmembers(n, g):
    u = torch.rand(5, 3, 3, generator=g, device=DEV, dtype=torch.float64)
    b = torch.arange(n, device=DEV, dtype=torch.float64)
    mu, sd, a = u[..., 0:1] * n, (5 + 25 * u[..., 1:2]) * n / 224, 0.2 + 0.8 * u[..., 2:3]
    return (a * torch.exp(-((b - mu) ** 2) / (2 * sd * sd))).sum(1)


def _scene(N, E, noise, g):
    A = -torch.log1p(-torch.rand(N, 5, generator=g, device=DEV, dtype=torch.float64))
    A = A / A.sum(1, keepdim=True)
    return A @ E + noise * torch.randn(N, E.shape[1], generator=g, device=DEV, dtype=torch.float64)


def _images(N, side, g):
    s = side / 64.0
    c = (16 + 32 * torch.rand(N, 2, generator=g, device=DEV, dtype=torch.float64)) * s
    u = torch.arange(side, device=DEV, dtype=torch.float64)
    gx = torch.exp(-((u - c[:, 0:1]) ** 2) / (2 * (4 * s) ** 2))
    gy = torch.exp(-((u - c[:, 1:2]) ** 2) / (2 * (4 * s) ** 2))
    return (gy[:, :, None] * gx[:, None, :]).reshape(N, side * side)


def _points(case, g):
    if case["data"] == "images":
        return _store(_images(case["N"], case["side"], g), "f32")
    if case["data"] == "scene":
        X = _scene(case["N"], _endmembers(case["n"], g), case["noise"], g)
    else:
        X = _curve(case["N"], case["n"], case["noise"], g)
    return _store(X, case["dtype"])


def _basis(n, k, seed):
    """A start: Q factor of a seeded Gaussian, rows = basis vectors, on the
    host, as a program that reads it from a file or draws it has it."""
    G = np.random.Generator(np.random.PCG64(seed)).standard_normal((n, k))
    Q, R = np.linalg.qr(G)
    return np.ascontiguousarray((Q * np.where(np.diag(R) < 0, -1.0, 1.0)).T)


def _batch_sizes(case):
    B, lo, hi = case["B"], math.log(case["N_min"]), math.log(case["N_max"])
    return [int(math.exp(lo + (hi - lo) * (b + 0.5) / B)) for b in range(B)]


def _inputs(case, seed):
    """(points, start): one tensor and one basis, or for a batch lists."""
    g, kind = _gen(seed), case["kind"]
    if kind == "batch":
        E = _endmembers(case["n"], g)
        Xs = [_store(_scene(N, E, 0.01, g), "bf16") for N in _batch_sizes(case)]
        return Xs, [_basis(case["n"], case["k"], seed + b) for b in range(case["B"])]
    if kind == "subsets":
        X = _store(_scene(case["N"], _endmembers(case["n"], g), 0.01, g), "f32")
        idx = torch.stack([torch.sort(torch.randperm(case["N"], generator=g, device=DEV)[:case["m"]])[0]
                           for _ in range(case["R"])])
        return (X, idx), _basis(case["n"], case["kmax"], seed)
    X = _points(case, g)
    return X, _basis(X.shape[1], case["kmax"] if kind == "sweep" else case["k"], seed)


def prepare(case, seed):
    kind = case["kind"]
    X, U = _inputs(case, seed)
    torch.cuda.synchronize()
    st = dict(case=case, U=U)
    if kind == "batch":
        st["sap"] = SapBatch([x.view(torch.uint16).cpu().numpy() for x in X], dtype=BF16)
        st["sap"].set_min_secant_length(case["eps"])
        return st
    if kind == "subsets":
        st["sap"] = SapBatch.from_subsamples(X[0].cpu().numpy(), X[1].cpu().numpy())
        return st
    sap = st["sap"] = Sap(X)
    if kind in ("run", "step"):
        sap.set_path(case["path"])
        sap.set_update_mode(case["mode"])
        if case["path"] == "restructured":
            sap.set_split(case["split"])
        if case["eps"] > 0:
            sap.set_min_secant_length(case["eps"])
    if kind in ("ascent", "threshold"):
        sap.set_basis(U)
    if kind == "softmin":
        st["U"] = torch.from_numpy(U).to(DEV)
    return st


def run(st):
    case, sap, U = st["case"], st["sap"], st["U"]
    kind = case["kind"]
    if kind == "run":
        sap.set_basis(U)
        hist, pairs = sap.run(case["alpha"], case["T"])
        return dict(ratios=hist, pairs=pairs, basis=sap.get_basis())
    if kind == "step":
        sap.set_basis(U)
        i, j, r = sap.step(case["alpha"])
        return dict(ratios=r, pairs=[i, j], basis=sap.get_basis())
    if kind == "batch":
        for b, Ub in enumerate(U):
            sap.set_basis(b, Ub)
        hist, pairs = sap.run(case["alpha"], case["T"])
        return dict(ratios=hist, pairs=pairs, basis=[sap.get_basis(b) for b in range(case["B"])])
    if kind == "sweep":
        k, ratios = sap.estimate_dim(U, case["T"], case["alpha"], case["threshold"])
        return dict(k=k, ratios=ratios, basis=sap.sweep_basis(case["kmax"]))
    if kind == "subsets":
        got = [sap.estimate_dim(b, U, case["T"], case["alpha"], case["threshold"]) for b in range(case["R"])]
        return dict(k=[k for k, _ in got], ratios=[r for _, r in got])
    if kind == "softmin":
        V = U.detach().requires_grad_(True)
        L = softmin(V, sap, case["tau"])
        L.backward()
        return dict(value=L.detach(), grad=V.grad)
    if kind == "ascent":
        sap.set_basis(U)
        hist = sap.softmin_ascent(case["tau"], case["eta"], case["T"])
        return dict(values=hist, basis=sap.get_basis())
    if kind == "pca":
        basis, sigma = sap.secant_pca(case["k"])
        return dict(basis=basis, sigma=sigma)
    sap.set_min_secant_length(case["eps"])
    i, j, r = sap.min_secant()
    return dict(pairs=[i, j], ratios=r, excluded=sap.stats()["n_excluded"])


# ------------------------------------------------------------------- work --

def work(case):
    """Bytes: the points and the bases in, the results out, once each.
    Flops: per evaluation the projection of the points (2 N n k) and per pair
    the projected difference, its square and the ratio (3 k + 2); the plain
    form projects every secant itself (2 n k + 3 n per pair); lengths, where
    the call forms them, 3 n per pair."""
    kind = case["kind"]
    if kind == "batch":
        Ns, n, k, T = _batch_sizes(case), case["n"], case["k"], case["T"]
        pts, pairs = sum(Ns), sum(N * (N - 1) // 2 for N in Ns)
        return dict(bytes=pts * n * 2 + case["B"] * 16 * n * k,
                    flops=(T + 1) * (2.0 * pts * n * k + pairs * (3 * k + 2)))
    if kind in ("sweep", "subsets"):
        n, R = (case["side"] ** 2, 1) if kind == "sweep" else (case["n"], case["R"])
        N = case["N"] if kind == "sweep" else case["m"]
        K, P = case["kmax"] * (case["kmax"] + 1) // 2, N * (N - 1) // 2
        return dict(bytes=R * N * n * 4 + 8 * n * case["kmax"],
                    flops=R * (case["T"] + 1) * (2.0 * N * n * K + P * (3.0 * K + 2 * case["kmax"])))
    N, n, k = case["N"], case["n"], case["k"]
    P = N * (N - 1) // 2
    size = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
    bytes_ = N * n * size + 16 * n * k
    if kind in ("run", "step"):
        per = P * (2.0 * n * k + 3 * n) if case["path"] == "plain" else 2.0 * N * n * k + P * (3.0 * k + 2)
        return dict(bytes=bytes_, flops=(case["T"] + (kind == "run")) * per)
    if kind == "softmin":  # value, then weights and their products with the differences
        return dict(bytes=bytes_, flops=4.0 * N * n * k + P * (3.0 * k + 6) + P * (7.0 * k + 8))
    if kind == "ascent":
        return dict(bytes=bytes_, flops=case["T"] * (4.0 * N * n * k + P * (10.0 * k + 14)) + P * (3.0 * k + 6))
    if kind == "pca":  # lengths, weighted differences per point, their Gram matrix, eigenvectors
        return dict(bytes=bytes_, flops=P * 3.0 * n + P * 5.0 * n + 2.0 * N * n * n + 10.0 * n ** 3)
    return dict(bytes=bytes_, flops=P * 3.0 * n + 2.0 * N * n * k + P * (3.0 * k + 2))


# ------------------------------------------------------- 64-bit reference --

class _Pairs:
    """Squared lengths of all pairs i < j in FP64, in blocks of rows against
    the columns from the block's first row on."""

    def __init__(self, X, eps=0.0):
        self.X = X.to(torch.float64)
        N, n = self.X.shape
        self.norm = float(self.X.norm(dim=1).max())
        self.blocks, self.excluded = [], 0
        cols = self.X.T.contiguous()
        for i0 in range(0, N, 2048):
            i1 = min(N, i0 + 2048)
            d2 = torch.zeros(i1 - i0, N - i0, dtype=torch.float64, device=X.device)
            for l in range(n):
                D = cols[l, i0:i1, None] - cols[l, None, i0:]
                d2.addcmul_(D, D)
            upper = torch.ones_like(d2, dtype=torch.bool).triu_(1)
            drop = upper & ((d2 == 0) | (d2 < eps * eps))
            self.excluded += int(drop.sum())
            d2[~upper | drop] = math.nan  # pairs that do not count
            self.blocks.append((i0, i1, d2))

    def squares(self, Y, i0, i1):
        q = torch.zeros(i1 - i0, Y.shape[0] - i0, dtype=torch.float64, device=Y.device)
        for c in range(Y.shape[1]):
            D = Y[i0:i1, c, None] - Y[None, i0:, c]
            q.addcmul_(D, D)
        return q

    def worst(self, U):
        """The pair with the smallest ratio under U (k, n), and the ratio:
        every pair within the rounding of Y = X U decided from explicit
        differences."""
        Y, best = self.X @ U.T, None
        for i0, i1, d2 in self.blocks:
            r = torch.nan_to_num((self.squares(Y, i0, i1) / d2).sqrt_(), nan=math.inf)
            m = float(r.min())
            if not math.isfinite(m) or (best and m > best[0] * (1 + 1e-6) + 1e-12):
                continue
            at = torch.nonzero(r <= m * (1 + 1e-6) + 1e-13)[:100000]
            D = self.X[at[:, 0] + i0] - self.X[at[:, 1] + i0]
            rr = (D @ U.T).norm(dim=1) / D.norm(dim=1)
            w = int(rr.argmin())
            if best is None or float(rr[w]) < best[0]:
                best = (float(rr[w]), int(at[w, 0]) + i0, int(at[w, 1]) + i0)
        return best

    def softmin(self, U, tau, grad=True):
        Y = self.X @ U.T
        rs = [(i0, i1, (self.squares(Y, i0, i1) / d2).sqrt_()) for i0, i1, d2 in self.blocks]
        parts = [torch.logsumexp(torch.nan_to_num(-r / tau, nan=-math.inf).reshape(-1), 0) for _, _, r in rs]
        L = -tau * float(torch.logsumexp(torch.stack(parts), 0))
        if not grad:
            return L, None
        z = torch.zeros_like(Y)
        for (i0, i1, r), (_, _, d2) in zip(rs, self.blocks):
            c = torch.nan_to_num(torch.exp((L - r) / tau) / (d2 * r), nan=0.0, posinf=0.0)
            z[i0:i1] += c.sum(1, keepdim=True) * Y[i0:i1] - c @ Y[i0:]
            z[i0:] += c.sum(0)[:, None] * Y[i0:] - c.T @ Y[i0:i1]
        return L, z.T @ (self.X - self.X.mean(0))


def _gram_schmidt(rows):
    out = []
    for v in rows:
        v = v.copy()
        for q in out:
            v -= (q @ v) * q
        nv = np.linalg.norm(v)
        out.append(v / nv if nv > 0 else v)
    return np.array(out)


def _rotate(U, s, alpha, mode):
    """Pivot, Gram-Schmidt, rotation of the first column (Algorithm 1)."""
    c = U @ s
    v = U.T @ c
    e = s - v
    t = int(np.argmax(np.abs(c)))
    Q = _gram_schmidt([v] + [U[l] for l in range(len(U)) if l != t])
    if mode == "angle":
        first = (1 - alpha) * v / np.linalg.norm(v) + alpha * e / np.linalg.norm(e)
    else:
        first = (1 - alpha) * v + alpha * e
    return _gram_schmidt([first / np.linalg.norm(first)] + list(Q[1:]))


def _trajectory(pairs, U, alpha, T, mode, last=True):
    hist, am, U = [], [], U.copy()
    for it in range(T + (1 if last else 0)):
        r, i, j = pairs.worst(torch.from_numpy(U).to(pairs.X.device))
        hist.append(r)
        am.append([i, j])
        if it < T:
            D = (pairs.X[i] - pairs.X[j]).cpu().numpy()
            U = _rotate(U, D / np.linalg.norm(D), alpha, mode)
    return np.array(hist), np.array(am, dtype=np.int64), U


def _exact_pca(X, k):
    X = X.to(torch.float64)
    N, n = X.shape
    C = torch.zeros(n, n, dtype=torch.float64, device=X.device)
    step = max(1, (1 << 27) // (N * n))
    for i0 in range(0, N, step):
        i1 = min(N, i0 + step)
        D = X[i0:i1, None, :] - X[None, i0:, :]
        d2 = (D * D).sum(2)
        keep = torch.ones_like(d2, dtype=torch.bool).triu_(1) & (d2 > 0)
        D = D * torch.where(keep, d2.clamp_min(1e-300).rsqrt(), 0.0)[:, :, None]
        D = D.reshape(-1, n)
        C += D.T @ D
    lam, V = np.linalg.eigh(C.cpu().numpy())
    V = V[:, ::-1][:, :k].T.copy()
    for v in V:
        v *= 1.0 if v[np.argmax(np.abs(v))] > 0 else -1.0
    return dict(basis=V, sigma=np.sqrt(lam[::-1][:k]))


def exact(case, seed):
    kind = case["kind"]
    # A free-running trajectory multiplies last-place differences by up to
    # ten per iteration (the update divides by the minimum ratio, which
    # starts near zero): after more than a few iterations the 64-bit
    # trajectory is no longer the value the one in the data's precision
    # approximates.
    if kind in ("run", "batch", "sweep", "subsets") and case["T"] > (4 if case.get("data") == "curve" else 8):
        return None
    X, U = _inputs(case, seed)
    if kind in ("run", "step"):
        p = _Pairs(X, case["eps"])
        h, am, V = _trajectory(p, U, case["alpha"], case["T"], case["mode"], last=kind == "run")
        return dict(ratios=h if kind == "run" else float(h[0]), pairs=am if kind == "run" else [int(a) for a in am[0]],
                    basis=V)
    if kind == "batch":
        got = [_trajectory(_Pairs(x, case["eps"]), u, case["alpha"], case["T"], "literal") for x, u in zip(X, U)]
        return dict(ratios=np.stack([h for h, _, _ in got]), pairs=np.stack([a for _, a, _ in got]),
                    basis=[V for _, _, V in got])
    if kind in ("sweep", "subsets"):
        # the bases of one and two columns meet near-ties at the size of
        # 64-bit rounding: their ratios stand among the others only by size
        sets = [X] if kind == "sweep" else [X[0][i] for i in X[1]]
        ratios, last = [], None
        for x in sets:
            p = _Pairs(x)
            tr = [_trajectory(p, U[:k], case["alpha"], case["T"], "literal") for k in range(1, case["kmax"] + 1)]
            ratios.append(np.array([h[-1] for h, _, _ in tr]))
            last = tr[-1][2]
        ks = [next((k + 1 for k, r in enumerate(q) if r > case["threshold"]), -1) for q in ratios]
        return dict(k=ks[0], ratios=ratios[0], basis=last) if kind == "sweep" else dict(k=ks, ratios=ratios)
    if kind == "softmin":
        L, G = _Pairs(X).softmin(torch.from_numpy(U).to(X.device), case["tau"])
        return dict(value=torch.tensor(L, dtype=torch.float64), grad=G)
    if kind == "ascent":
        p, V, hist = _Pairs(X), torch.from_numpy(U).to(X.device), []
        for _ in range(case["T"]):
            L, G = p.softmin(V, case["tau"])
            hist.append(L)
            G = G - (G @ V.T) @ V
            V = torch.from_numpy(_gram_schmidt((V + case["eta"] * G / G.norm()).cpu().numpy())).to(X.device)
        hist.append(p.softmin(V, case["tau"], grad=False)[0])
        return dict(values=np.array(hist), basis=V.cpu().numpy())
    if kind == "pca":
        return _exact_pca(X, case["k"])
    p = _Pairs(X, case["eps"])
    r, i, j = p.worst(torch.from_numpy(U).to(X.device))
    return dict(pairs=[i, j], ratios=r, excluded=p.excluded)
