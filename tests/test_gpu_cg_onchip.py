"""The one-launch CG filter (vectors on the chip) at the edges of its split: signals around
multiples of the piece a CTA owns, shorter than the window, with the smallest and largest
radius and every weight mode; images of one pixel to several rectangles with ragged edges.
Against the oracle's Algorithm 2, with coefficients, early stops and the smallest kmax.

A system of n unknowns is run for at most n / 3 steps: past convergence to rounding the
recurrence divides rounding errors by each other, on any path.

Bounds: the repository's 1e-5 (FP32) and 1e-11 (FP64) bars for filter outputs; the recorded
alpha and beta carry the error of a quotient of FP32 sums (1e-4) or FP64 sums (1e-9)."""
import numpy as np
import pytest
import torch

from oracle import solvers
from oracle.graph import Graph
from paper_1509_02468_gb300 import synth
from tests.gpu_helpers import TOL_F32, TOL_F64, bf, host, rel_l2

pytestmark = pytest.mark.gpu


def _signal(n, dtype):
    rng = np.random.default_rng(n)
    x = np.repeat(rng.uniform(0, 1, (n + 39) // 40), 40)[:n] + 0.1 * rng.standard_normal(n)
    return torch.as_tensor(x, device="cuda").to(dtype)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n,radius", [(2, 1), (7, 5), (64, 5), (65, 5), (127, 32), (1000, 1), (4097, 5), (9473, 7),
                                      (30001, 5)])
def test_signals(n, radius, dtype):
    x0 = _signal(n, dtype)
    G = bf().bf_weights(x0, radius, 3.0, 0.1)
    O = Graph(host(x0), (1, n), radius, 3.0, 0.1)
    for kw in ({}, {"shift": 0.1}, {"precond": "identity"}):
        iters = min(6, max(1, n // 3))
        x, info, hist = bf().cg_filter(G, x0, iters, hist=True, **kw)
        ref = solvers.cg(O, host(x0), iters, **kw)
        assert info.iters == ref["iters"]
        assert rel_l2(host(x), ref["x"]) < (TOL_F64 if dtype == torch.float64 else TOL_F32)
        if n > 64:
            h = hist.cpu().numpy().reshape(-1, 2)
            tol = 1e-9 if dtype == torch.float64 else 1e-4
            np.testing.assert_allclose(h[:, 0], ref["alpha"], rtol=tol)
            np.testing.assert_allclose(h[1:, 1], ref["beta"][1:], rtol=tol)


@pytest.mark.parametrize("mode", ["stored_f32", "stored_bf16"])
def test_signals_with_stored_weights(mode):
    x0 = _signal(3001, torch.float32)
    G = bf().bf_weights(x0, 5, 3.0, 0.1, weight_mode=mode)
    O = Graph.from_taps(host(bf().graph_export_weights(G)), (1, 3001), 5)
    x, _, _ = bf().cg_filter(G, x0, 8)
    assert rel_l2(host(x), solvers.cg(O, host(x0), 8)["x"]) < TOL_F32


@pytest.mark.parametrize("shape", [(1, 1), (2, 3), (4, 32), (5, 33), (37, 31), (97, 131), (130, 64), (203, 517)])
def test_images(shape):
    rng = np.random.default_rng(shape[1])
    img = (synth.polygon_image(*shape, seed=5, polygons=6)[1] if min(shape) > 8
           else rng.uniform(0, 1, shape).astype(np.float32))
    g = torch.as_tensor(img, device="cuda")
    G = bf().bf_weights(g, 3, 2.0, 0.08)
    O = Graph(img.astype(np.float64), shape, 3, 2.0, 0.08)
    x0 = g.reshape(-1)
    for kw in ({}, {"shift": 0.05}, {"precond": "identity", "beta": "printed"}):
        okw = dict(kw)
        if "beta" in okw:
            okw["beta"] = "ss"
        iters = min(7, max(1, img.size // 3))
        x, info, hist = bf().cg_filter(G, x0, iters, hist=True, **kw)
        ref = solvers.cg(O, host(x0), iters, **okw)
        assert rel_l2(host(x), ref["x"]) < TOL_F32
        assert info.iters == ref["iters"]
        if img.size > 100:
            np.testing.assert_allclose(hist.cpu().numpy()[0::2], ref["alpha"], rtol=1e-4)
    y = x0.clone()                                          # in place, and no iteration at all
    bf().cg_filter(G, y, iters, out=y)
    assert rel_l2(host(y), solvers.cg(O, host(x0), iters)["x"]) < TOL_F32
    assert torch.equal(bf().cg_filter(G, x0, 0)[0], x0)


def test_early_stop_and_streams():
    """A tolerance stops the launch at the oracle's iteration; runs on two graphs and two
    streams at once give what they give alone."""
    img = synth.polygon_image(180, 301, seed=6, polygons=6)[1]
    g = torch.as_tensor(img, device="cuda")
    G, G2 = bf().bf_weights(g, 3, 2.0, 0.08), bf().bf_weights(g.t().contiguous(), 3, 2.0, 0.08)
    O = Graph(img.astype(np.float64), img.shape, 3, 2.0, 0.08)
    x0, x1 = g.reshape(-1), g.t().contiguous().reshape(-1)
    x, info, _ = bf().cg_filter(G, x0, 400, shift=0.5, tol=1e-3)
    ref = solvers.cg(O, host(x0), 400, shift=0.5, tol=1e-3)
    assert info.status == "converged" and info.iters == ref["iters"]
    assert rel_l2(host(x), ref["x"]) < TOL_F32
    a, b = bf().cg_filter(G, x0, 15)[0], bf().cg_filter(G2, x1, 15)[0]
    s, t = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    oa, ob = torch.empty_like(x0), torch.empty_like(x1)
    for _ in range(3):
        bf().cg_filter(G, x0, 15, out=oa, sync=False, stream=s)
        bf().cg_filter(G2, x1, 15, out=ob, sync=False, stream=t)
    torch.cuda.synchronize()
    assert torch.equal(a, oa) and torch.equal(b, ob)


@pytest.mark.parametrize("radius", [1, 2, 3])
@pytest.mark.parametrize("shape", [(3, 4), (5, 33), (40, 61), (66, 130)])
def test_guided_images(shape, radius):
    from oracle.guided import GuidedGraph
    img = np.random.default_rng(radius).uniform(0, 1, shape)
    img[:, shape[1] // 2:] *= 0.3
    g = torch.as_tensor(img.astype(np.float32), device="cuda")
    G = bf().guided_graph(g, radius, 0.01)
    O = GuidedGraph(host(g), shape, radius, 0.01)
    iters = min(7, max(1, img.size // 4))
    for kw in ({}, {"shift": 0.5}, {"precond": "identity"}):
        x, info, _ = bf().cg_filter(G, g.reshape(-1), iters, **kw)
        ref = solvers.cg(O, host(g).reshape(-1), iters, **kw)
        assert info.iters == ref["iters"]
        assert rel_l2(host(x), ref["x"]) < TOL_F32


@pytest.mark.parametrize("shape", [(1103, 1201), (1290, 1002), (1030, 1280), (601, 2203)])
def test_images_beyond_the_chip(shape):
    """Images too large for the one-launch form, with rows that are padded to whole vectors and
    rows that are not, against the FP64 path on the same guide (itself held to the oracle)."""
    rng = np.random.default_rng(shape[1])
    img = np.cumsum(rng.uniform(-0.03, 0.03, shape), axis=1).astype(np.float32)
    g = torch.as_tensor(img, device="cuda")
    G, G64 = bf().bf_weights(g, 3, 2.0, 0.08), bf().bf_weights(g.double(), 3, 2.0, 0.08)
    x0 = g.reshape(-1)
    for kw in ({}, {"shift": 0.05, "precond": "identity"}):
        ref = bf().cg_filter(G64, x0.double(), 6, **kw)[0]
        x, info, _ = bf().cg_filter(G, x0, 6, **kw)
        assert info.iters == 6 and rel_l2(host(x), host(ref)) < TOL_F32
        y = x0.clone()
        bf().cg_filter(G, y, 6, out=y, **kw)
        assert torch.equal(x, y)
    wide = torch.zeros(x0.numel() + 1, device="cuda")        # vectors off the 16-byte grid
    wide[1:] = x0
    out = torch.empty_like(wide)[1:]
    bf().cg_filter(G, wide[1:], 6, out=out)
    assert rel_l2(host(out), host(bf().cg_filter(G64, x0.double(), 6)[0])) < TOL_F32


@pytest.mark.parametrize("kind,shape", [("image", (64, 64)), ("image", (63, 97)), ("image", (128, 128)), ("image", (130, 161)),
                                        ("guided", (128, 128)), ("signal", (9472,)), ("signal", (9473,)), ("signal", (18944,)),
                                        ("signal", (18945,))])
def test_splits_that_leave_room_for_other_streams(kind, shape):
    """Small images by rectangles of four units and mid-length signals by pieces of 256 samples:
    either side of the lines where those splits are taken, alone and four at a time."""
    n = int(np.prod(shape))
    if kind == "signal":
        x0 = _signal(n, torch.float32)
        G = [bf().bf_weights(x0, 5, 3.0, 0.1) for _ in range(4)]
        O = Graph(host(x0), (1, n), 5, 3.0, 0.1)
    else:
        from oracle.guided import GuidedGraph
        g = torch.as_tensor(synth.polygon_image(*shape, seed=7, polygons=6)[1].astype(np.float32), device="cuda")
        x0 = g.reshape(-1).clone()
        G = [bf().guided_graph(g, 2, 0.01) if kind == "guided" else bf().bf_weights(g, 3, 2.0, 0.08) for _ in range(4)]
        O = (GuidedGraph(host(g), shape, 2, 0.01) if kind == "guided" else Graph(host(g), shape, 3, 2.0, 0.08))
    ref = solvers.cg(O, host(x0).reshape(-1), 12, shift=0.2)["x"]
    x, info, _ = bf().cg_filter(G[0], x0, 12, shift=0.2)
    assert info.iters == 12 and rel_l2(host(x), ref) < TOL_F32
    streams = [torch.cuda.Stream() for _ in G]
    outs = [torch.empty_like(x0) for _ in G]
    torch.cuda.synchronize()
    for _ in range(3):
        for H, o, s in zip(G, outs, streams):
            bf().cg_filter(H, x0, 12, shift=0.2, out=o, sync=False, stream=s)
    torch.cuda.synchronize()
    for o in outs:
        assert torch.equal(o, x)


def test_small_runs_on_eight_streams_overlap():
    """Eight runs on eight streams take far less than eight runs (they would one after the other)."""
    import time
    g = torch.as_tensor(synth.polygon_image(128, 128, seed=8, polygons=6)[1].astype(np.float32), device="cuda")
    x0 = g.reshape(-1)
    G = [bf().bf_weights(g, 3, 2.0, 0.08) for _ in range(8)]
    streams, outs = [torch.cuda.Stream() for _ in G], [torch.empty_like(x0) for _ in G]

    def run(k):
        times = []
        for _ in range(7):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for i in range(k):
                bf().cg_filter(G[i], x0, 300, shift=0.01, out=outs[i], sync=False, stream=streams[i])
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t)
        return sorted(times)[3]

    assert run(8) < 5.0 * run(1)
