"""The calls a user of this framework makes, as measurable cases.

Every case goes through the public binding (``paper_1509_02468_gb300.bf``) the way a
denoising program does: graphs and blocks are prepared once, then filters, operator
applications, graph updates or training gradients run on them.  The workloads are the
repository's configurations (the 4096-sample FP64 signal; the 7 x 7 window images at
sigma_s 2, sigma_r 0.08; the mixed batch; the learned preconditioner) and generic image
sizes, ragged ones among them.  ``exact`` restates each in FP64 with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1509_02468_gb300 import bf

SIGMA_S, SIGMA_R = 2.0, 0.08           # the image workloads' widths (7 x 7 window)
SIG_S, SIG_R = 3.0, 0.1                # the signal workloads' widths (11 taps)
NET_SHIFT = 1e-2                       # sigma of the training pairs' system


def listed():
    return [
        # the smallest call: one FP64 signal through the CG filter (launch latency)
        {"name": "cg_signal_4096_f64", "kind": "cg_signal", "n": 4096, "dtype": "f64", "iters": 20},
        # the next frame of a full-HD stream: weights and degree of a new guide
        {"name": "weights_1080x1920", "kind": "weights", "ny": 1080, "nx": 1920},
        # the benchmark image through the CG filter
        {"name": "cg_image_512", "kind": "cg_image", "ny": 512, "nx": 512, "iters": 50,
         "precond": "jacobi", "shift": 0.0},
        # a large photograph of odd size through the CG filter
        {"name": "cg_image_1531x2047", "kind": "cg_image", "ny": 1531, "nx": 2047, "iters": 50,
         "precond": "jacobi", "shift": 0.0},
        # the benchmark image through the block filter (the framework's main call)
        {"name": "lobpcg_image_512_k16", "kind": "lobpcg_image", "ny": 512, "nx": 512, "k": 16,
         "iters": 30},
        # the operator alone on a block, as a user's own block eigensolver calls it
        {"name": "apply_2048_k16", "kind": "apply", "ny": 2048, "nx": 2048, "k": 16,
         "mode": "onthefly"},
        # the operator on one vector with FP32 weights stored (the HBM-bound form)
        {"name": "apply_2048_k1_f32w", "kind": "apply", "ny": 2048, "nx": 2048, "k": 1,
         "mode": "stored_f32"},
        # the precision study's operator: BF16 weights stored, a block of vectors
        {"name": "apply_1024_k16_bf16w", "kind": "apply", "ny": 1024, "nx": 1024, "k": 16,
         "mode": "stored_bf16"},
        # the nonlinear bilateral iteration on an odd-sized image
        {"name": "reguided_767x1021", "kind": "reguided", "ny": 767, "nx": 1021, "iters": 10},
        # the guided filter's graph through the CG filter
        {"name": "guided_cg_512", "kind": "guided_cg", "ny": 512, "nx": 512, "radius": 2,
         "iters": 50},
        # a server's mixed batch: uneven images and signals in one call
        {"name": "batch_cg_64", "kind": "batch_cg", "images": 48, "signals": 16, "iters": 20,
         "pick": 4},
        # one training step of the learned preconditioner: forward, backward, gradient
        {"name": "net_train_256", "kind": "net_train", "side": 256, "pairs": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cg_signal", "weights", "cg_image", "lobpcg_image", "apply", "reguided",
                       "guided_cg", "batch_cg", "net_train"])
    if kind == "cg_signal":
        return {"kind": kind, "n": _log(rng, 1000, 200000), "dtype": rng.choice(["f64", "f64", "f32"]),
                "iters": rng.choice([10, 20, 30])}
    if kind == "weights":
        return {"kind": kind, "ny": _log(rng, 128, 2048), "nx": _log(rng, 128, 2048)}
    if kind == "cg_image":
        return {"kind": kind, "ny": _log(rng, 128, 1600), "nx": _log(rng, 128, 1600),
                "iters": rng.choice([20, 50]), "precond": rng.choice(["jacobi", "jacobi", "identity"]),
                "shift": rng.choice([0.0, 0.0, 0.01])}
    if kind == "lobpcg_image":
        return {"kind": kind, "ny": _log(rng, 256, 512), "nx": _log(rng, 256, 512),
                "k": rng.choice([8, 16]), "iters": rng.choice([10, 20])}
    if kind == "apply":
        return {"kind": kind, "ny": _log(rng, 128, 2000), "nx": _log(rng, 128, 2000),
                "k": rng.choice([1, 4, 8, 16]),
                "mode": rng.choice(["onthefly", "onthefly", "stored_f32", "stored_bf16"])}
    if kind == "reguided":
        return {"kind": kind, "ny": _log(rng, 128, 2000), "nx": _log(rng, 128, 2000),
                "iters": rng.choice([5, 10, 20])}
    if kind == "guided_cg":
        return {"kind": kind, "ny": _log(rng, 128, 700), "nx": _log(rng, 128, 700),
                "radius": rng.choice([1, 2, 3]), "iters": rng.choice([20, 50])}
    if kind == "batch_cg":
        return {"kind": kind, "images": rng.randint(8, 48), "signals": rng.randint(4, 16),
                "iters": rng.choice([10, 20]), "pick": rng.randint(0, 1 << 20)}
    return {"kind": kind, "side": _log(rng, 96, 320), "pairs": rng.randint(2, 8)}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _image(ny, nx, seed, noise=0.05):
    """A gradient with 20 star-shaped patches of flat level and Gaussian noise (float32)."""
    rng = np.random.default_rng(seed)
    side = float(max(nx, ny))
    ys = torch.arange(ny, device="cuda", dtype=torch.float32).add_(0.5).view(-1, 1)
    xs = torch.arange(nx, device="cuda", dtype=torch.float32).add_(0.5).view(1, -1)
    a, b = rng.uniform(0.0, 1.0, 2)
    ang = rng.uniform(0.0, 2.0 * math.pi)
    img = a + b * 0.5 * (1.0 + (math.cos(ang) * xs + math.sin(ang) * ys) / side)
    for _ in range(20):
        cx, cy = rng.uniform(0.0, nx), rng.uniform(0.0, ny)
        rad, depth = rng.uniform(0.05, 0.25) * side, rng.uniform(0.0, 0.5)
        lobes, turn = int(rng.integers(3, 9)), rng.uniform(0.0, 2.0 * math.pi)
        dx, dy = xs - cx, ys - cy
        edge = rad * (1.0 - depth * torch.cos(lobes * torch.atan2(dy, dx) + turn))
        img = torch.where(dx * dx + dy * dy < edge * edge, float(rng.uniform(0.0, 1.0)), img)
    return (img + noise * torch.randn((ny, nx), device="cuda", generator=_gen(seed + 1))).contiguous()


def _signal(n, seed, dtype, noise=0.1):
    """12 constant pieces (levels U[0, 1]) and Gaussian noise."""
    rng = np.random.default_rng(seed)
    edges = np.sort(rng.choice(np.arange(1, n), size=11, replace=False))
    clean = rng.uniform(0.0, 1.0, 12)[np.searchsorted(edges, np.arange(n), side="right")]
    return torch.as_tensor(clean + noise * rng.standard_normal(n), device="cuda").to(dtype)


def _shapes(case):
    """(ndim, ny, nx) of a mixed batch: sides log-uniform in [64, 512], lengths in [1e3, 2e5]."""
    rng = np.random.default_rng(case["pick"])
    side = lambda: int(round(math.exp(rng.uniform(math.log(64), math.log(512)))))  # noqa: E731
    out = [(2, side(), side()) for _ in range(case["images"])]
    return out + [(1, 1, int(round(math.exp(rng.uniform(math.log(1e3), math.log(2e5))))))
                  for _ in range(case["signals"])]


def _batch_inputs(case, seed):
    return [_image(ny, nx, 1000 * seed + i) if nd == 2 else _signal(nx, 1000 * seed + i, torch.float32)
            for i, (nd, ny, nx) in enumerate(_shapes(case))]


def _block(guide, k, seed):
    """Column 0 the image, the others N(0, 1)."""
    X = torch.randn((guide.numel(), k), device="cuda", generator=_gen(seed + 2))
    X[:, 0] = guide.reshape(-1)
    return X


def _net_weights(seed):
    """The Jacobi-equivalent start of the training (channels 0 and 1 carry the residual)
    with N(0, 0.05^2) on the other channels, as a net some steps into its training."""
    rng = np.random.default_rng(seed)
    W1 = 0.05 * rng.standard_normal((16, 3, 3, 3))
    W2 = 0.05 * rng.standard_normal((16, 16, 3, 3))
    W3 = 0.05 * rng.standard_normal((1, 16, 3, 3))
    W1[0:2] = W2[0:2] = W3[0, 0:2] = 0.0
    W1[0, 0, 1, 1], W1[1, 0, 1, 1] = 1.0, -1.0
    W2[0, 0, 1, 1], W2[1, 1, 1, 1] = 1.0, 1.0
    W3[0, 0, 1, 1], W3[0, 1, 1, 1] = 1.0, -1.0
    return [W1.astype(np.float32), W2.astype(np.float32), W3.astype(np.float32)]


def _net_pairs(case, seed):
    """(guide, [(r, z)]): z a smooth field plus noise, r = (L + sigma I) z."""
    side = case["side"]
    guide = _image(side, side, seed)
    op = _Operator(guide.double(), 3, SIGMA_S, SIGMA_R)
    pairs = []
    for j in range(case["pairs"]):
        z = torch.randn((1, 1, side, side), device="cuda", generator=_gen(seed + 10 + j)).double()
        for _ in range(3):
            z = torch.nn.functional.avg_pool2d(z, 5, stride=1, padding=2) * 2.0 + 0.1 * z
        z = z.view(side, side).float()
        r = (op.L(z.double()) + NET_SHIFT * z.double()).float()
        pairs.append((r.reshape(-1).contiguous(), z.reshape(-1).contiguous()))
    return guide, pairs


def prepare(case, seed):
    kind = case["kind"]
    if kind == "cg_signal":
        x = _signal(case["n"], seed, torch.float64 if case["dtype"] == "f64" else torch.float32)
        return case, bf.bf_weights(x, 5, SIG_S, SIG_R), x
    if kind == "batch_cg":
        xs = _batch_inputs(case, seed)
        graphs = [bf.bf_weights(x, 3, SIGMA_S, SIGMA_R) if x.dim() == 2 else bf.bf_weights(x, 5, SIG_S, SIG_R)
                  for x in xs]
        return case, bf.Batch(graphs), [x.reshape(-1) for x in xs]
    if kind == "net_train":
        guide, pairs = _net_pairs(case, seed)
        return case, bf.Net(_net_weights(seed)), bf.bf_weights(guide, 3, SIGMA_S, SIGMA_R), pairs
    img = _image(case["ny"], case["nx"], seed)
    if kind == "weights":                     # the stream's graph, made from an earlier frame
        return case, bf.bf_weights(_image(case["ny"], case["nx"], seed + 500), 3, SIGMA_S, SIGMA_R), img
    if kind == "guided_cg":
        return case, bf.guided_graph(img, case["radius"], 0.01), img.reshape(-1)
    g = bf.bf_weights(img, 3, SIGMA_S, SIGMA_R, weight_mode=case.get("mode", "onthefly"))
    if kind == "apply":
        return case, g, _block(img, case["k"], seed)
    if kind == "lobpcg_image":
        return case, g, _block(img, case["k"], seed)
    return case, g, img.reshape(-1)           # cg_image, reguided


def run(state):
    case, kind = state[0], state[0]["kind"]
    if kind in ("cg_signal", "guided_cg"):
        return bf.cg_filter(state[1], state[2], case["iters"], sync=False)[0]
    if kind == "cg_image":
        return bf.cg_filter(state[1], state[2], case["iters"], precond=case["precond"],
                            shift=case["shift"], sync=False)[0]
    if kind == "weights":
        return bf.graph_degree(bf.graph_update(state[1], state[2]))
    if kind == "lobpcg_image":                # the filtered image is the call's product
        return bf.lobpcg_filter(state[1], state[2], case["iters"], want_X=False, sync=False)["y"]
    if kind == "apply":
        return bf.bf_apply(state[1], "L", state[2])
    if kind == "reguided":
        out = bf.reguided_filter(state[1], state[2], case["iters"])
        return out, bf.graph_degree(state[1])
    if kind == "batch_cg":
        return state[1].cg(state[2], case["iters"], sync=False)[0]
    net, g = state[1], state[2]               # net_train: gradient and loss over the pairs
    net.zero_grad()
    for r, z in state[3]:
        net.accumulate(g, r, z)
    return net.grad()


# ---------------------------------------------------------------- what a pass needs
# operations per pixel: a tap of the difference form is 4 for the exponent, 1 exponential
# and 3 for the sum; pairs counted from both ends
TAP = 8


def work(case):
    kind = case["kind"]
    if kind == "cg_signal":
        n, es = case["n"], 8 if case["dtype"] == "f64" else 4
        return {"bytes": 3 * es * n, "flops": n * (case["iters"] + 1) * (10 * TAP + 16)}
    if kind == "batch_cg":
        it = case["iters"] + 1
        sh = _shapes(case)
        return {"bytes": 12 * sum(ny * nx for _, ny, nx in sh),
                "flops": sum(ny * nx * it * ((48 if nd == 2 else 10) * TAP + 16) for nd, ny, nx in sh)}
    if kind == "net_train":
        n, mac = case["side"] ** 2, 16 * 27 + 16 * 144 + 144
        return {"bytes": case["pairs"] * 8 * n + 8 * n, "flops": case["pairs"] * n * 6 * mac}
    n = case["ny"] * case["nx"]
    if kind == "weights":
        return {"bytes": 8 * n, "flops": n * 48 * 6}
    if kind == "cg_image":
        return {"bytes": 12 * n, "flops": n * (case["iters"] + 1) * (48 * TAP + 16)}
    if kind == "guided_cg":
        taps = 2 * (2 * case["radius"] + 1) ** 2
        return {"bytes": 20 * n, "flops": n * (case["iters"] + 1) * (4 * taps + 16)}
    if kind == "reguided":
        return {"bytes": 12 * n, "flops": n * case["iters"] * 48 * TAP}
    k = case["k"]
    if kind == "apply":
        wb = {"onthefly": 4, "stored_f32": 96, "stored_bf16": 48}[case["mode"]]
        return {"bytes": (wb + 8 * k) * n, "flops": n * 48 * (3 * k + (5 if wb == 4 else 0))}
    # LOBPCG: per iteration three block applies, two Gram matrices, the block updates
    return {"bytes": (4 + 4 + 4 * k + 4) * n,
            "flops": n * case["iters"] * (3 * 48 * (3 * k + 5) + 18 * k * k * 2 + 12 * k * k)}


# ---------------------------------------------------------------- the same in FP64
class _Operator:
    """The graph Laplacian of Eq. 2's weights on an FP64 image or signal, by shifted slices."""

    def __init__(self, guide, radius, sigma_s, sigma_r, rounded=None):
        g = guide.double()
        g = g.view(1, -1) if g.dim() == 1 else g
        self.shape = ny, nx = g.shape
        self.taps = []
        self.d = torch.ones_like(g)
        for dy in range(0, (radius if ny > 1 else 0) + 1):
            for dx in range(-radius, radius + 1):
                if (dy, dx) <= (0, 0) or dy >= ny or abs(dx) >= nx:
                    continue
                A = (slice(0, ny - dy), slice(max(0, -dx), nx - max(0, dx)))
                B = (slice(dy, ny), slice(max(0, dx), nx - max(0, -dx)))
                w = torch.exp(-(dx * dx + dy * dy) / (2 * sigma_s**2) - (g[A] - g[B]) ** 2 / (2 * sigma_r**2))
                if rounded is not None:
                    w = w.float().to(rounded).double()
                self.taps.append((A, B, w))
                self.d[A] += w
                self.d[B] += w

    def L(self, x):
        """x: [ny, nx] or [ny, nx, k]."""
        y = torch.zeros_like(x)
        for A, B, w in self.taps:
            t = (x[A] - x[B]) * (w if x.dim() == 2 else w.unsqueeze(-1))
            y[A] += t
            y[B] -= t
        return y


class _Guided:
    """The guided filter's Laplacian N x - N GF(x) (windows truncated at the border)."""

    def __init__(self, guide, r, eps):
        self.g, self.r = guide.double(), r
        self.d = self.box(torch.ones_like(self.g))
        self.mu = self.box(self.g) / self.d
        self.iv = 1.0 / (self.box(self.g * self.g) / self.d - self.mu**2 + eps)

    def box(self, v):
        p = 2 * self.r + 1
        ones = torch.ones((1, 1, p, p), dtype=torch.float64, device=v.device)
        return torch.nn.functional.conv2d(v[None, None], ones, padding=self.r)[0, 0]

    def L(self, x):
        m = self.box(x) / self.d
        a = (self.box(self.g * x) / self.d - self.mu * m) * self.iv
        return self.d * x - (self.box(a) * self.g + self.box(m - a * self.mu))


def _cg(op, x0, iters, precond="jacobi", shift=0.0):
    tinv = 1.0 / op.d if precond == "jacobi" else torch.ones_like(op.d)
    x, r, p, sr = x0.clone(), -op.L(x0), None, None
    for _ in range(iters):
        s = tinv * r
        sr_new = (s * r).sum()
        p = s if p is None else s + (s * (r - r_old)).sum() / sr * p
        q = op.L(p) + shift * p
        a = sr_new / (p * q).sum()
        x = x + a * p
        r_old, r, sr = r, r - a * q, sr_new
    return x


def _ritz(GA, GB, k):
    s = GB.diagonal().rsqrt()
    R = torch.linalg.cholesky(GB * s[:, None] * s[None, :])
    M = torch.linalg.solve_triangular(R, GA * s[:, None] * s[None, :], upper=False)
    M = torch.linalg.solve_triangular(R, M.T, upper=False)
    lam, V = torch.linalg.eigh(0.5 * (M + M.T))
    return lam[:k], torch.linalg.solve_triangular(R.T, V[:, :k], upper=True) * s[:, None]


def _lobpcg_y(op, X, iters):
    ny, nx = op.shape
    n, k = X.shape
    d = op.d.reshape(-1, 1)
    L = lambda V: op.L(V.view(ny, nx, -1)).reshape(n, -1)  # noqa: E731
    x0 = X[:, 0:1].clone()
    theta, C = _ritz(X.T @ L(X), X.T @ (d * X), k)
    X, P = X @ C, None
    for _ in range(iters):
        AX = L(X)
        W = (AX - d * X * theta) / d
        S = torch.cat([X, W] + ([P] if P is not None else []), 1)
        AS = torch.cat([AX, L(S[:, k:])], 1)
        theta, C = _ritz(S.T @ AS, S.T @ (d * S), k)
        X, P = S @ C, S[:, k:] @ C[k:]
        P = P - X @ (X.T @ (d * P))
    return (X @ (X.T @ (d * x0))).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "cg_signal":
        x = _signal(case["n"], seed, torch.float64 if case["dtype"] == "f64" else torch.float32)
        op = _Operator(x, 5, SIG_S, SIG_R)
        return _cg(op, x.double().view(1, -1), case["iters"]).reshape(-1)
    if kind == "batch_cg":
        out = []
        for x in _batch_inputs(case, seed):
            op = _Operator(x, 3, SIGMA_S, SIGMA_R) if x.dim() == 2 else _Operator(x, 5, SIG_S, SIG_R)
            out.append(_cg(op, x.double().view(op.shape), case["iters"]).reshape(-1))
        return out
    if kind == "net_train":
        guide, pairs = _net_pairs(case, seed)
        g, side = guide.double(), case["side"]
        d = _Operator(g, 3, SIGMA_S, SIGMA_R).d
        W = [torch.as_tensor(w, device="cuda").to(torch.bfloat16).double().requires_grad_() for w in _net_weights(seed)]
        conv = torch.nn.functional.conv2d
        loss = 0.0
        for r, z in pairs:
            c0, zz = r.double().view(side, side) / d, z.double().view(side, side)
            rho = (c0 * c0).mean().sqrt()
            h = torch.stack([c0 / rho, g, 1.0 / d])[None]
            h = conv(torch.relu(conv(torch.relu(conv(h, W[0], padding=1)), W[1], padding=1)), W[2], padding=1)
            loss = loss + ((rho * h[0, 0] - zz) ** 2).sum() / (zz * zz).sum()
        loss.backward()
        return np.concatenate([w.grad.cpu().numpy().ravel() for w in W]), float(loss)
    img = _image(case["ny"], case["nx"], seed)
    if kind == "guided_cg":
        return _cg(_Guided(img, case["radius"], 0.01), img.double(), case["iters"]).reshape(-1)
    if kind == "reguided":
        x = img.double()
        for _ in range(case["iters"]):
            op = _Operator(x, 3, SIGMA_S, SIGMA_R)
            x = x - op.L(x) / op.d
        return x.reshape(-1), op.d.reshape(-1)
    rounded = torch.bfloat16 if case.get("mode") == "stored_bf16" else None
    op = _Operator(img, 3, SIGMA_S, SIGMA_R, rounded)
    if kind == "weights":
        return op.d.reshape(-1)
    if kind == "cg_image":
        return _cg(op, img.double(), case["iters"], case["precond"], case["shift"]).reshape(-1)
    X = _block(img, case["k"], seed).double()
    if kind == "apply":
        return op.L(X.view(case["ny"], case["nx"], -1)).reshape(X.shape)
    return _lobpcg_y(op, X, case["iters"])
