"""Fixed-count runs of the one-launch CG filter past convergence: the residual's squares fall
below the range of a float (FP64: below that of alpha / s^T r) while the terms themselves are
still there, and x has to stay the solution it reached.

Bounds: the repository's 1e-5 (FP32) and 1e-11 (FP64) bars for filter outputs, against the
oracle's solution of (L + sigma I) x = sigma x0.  `may_end`: the run outlives its terms, where
p^T q = 0 is a breakdown on any path; otherwise it has to run through or to converge."""
import numpy as np
import pytest
import torch

from oracle import solvers
from oracle.graph import Graph
from oracle.guided import GuidedGraph
from paper_1509_02468_gb300 import synth
from tests.gpu_helpers import TOL_F32, TOL_F64, bf, host, rel_l2

pytestmark = pytest.mark.gpu


def _solution(O, x0, shift):
    ref = solvers.cg(O, host(x0), 3000, shift=shift, tol=1e-14)
    assert ref["status"] == "converged"
    return ref["x"]


def _check(G, x0, sol, tol, steps, may_end, **kw):
    x = bf().cg_filter(G, x0, steps, sync=False, **kw)[0]
    assert torch.isfinite(x).all() and rel_l2(host(x), sol) < tol
    try:
        y, info, hist = bf().cg_filter(G, x0, steps, hist=True, **kw)
    except bf().BFError as e:
        assert may_end and e.code == bf().BF_EBREAKDOWN
        return
    assert torch.equal(x, y)
    assert info.status == "converged" or info.iters == steps
    assert torch.isfinite(hist[:2 * info.iters]).all() and np.isfinite(info.rnorm)
    if G.n <= 1 << 18 and G.params.__class__.__name__ == "bf_params":
        z, zi = bf().cg_filter_noalloc(G, x0, steps, **kw)
        assert torch.equal(x, z) and zi.iters == info.iters


@pytest.mark.parametrize("scale", [1.0, 255.0])
@pytest.mark.parametrize("shape,shift,precond,steps,may_end", [
    ((200, 300), 1.0, "jacobi", 100, False), ((64, 64), 10.0, "jacobi", 50, False),
    ((64, 64), 1.0, "identity", 100, False), ((64, 64), 100.0, "identity", 17, False),
    ((64, 64), 100.0, "identity", 50, True), ((180, 301), 0.1, "jacobi", 280, False)])
def test_images(shape, shift, precond, steps, may_end, scale):
    """x0 also as 8-bit values (its scale is that of the sums)."""
    img = synth.polygon_image(*shape, 5, polygons=6)[1].astype(np.float32)
    g = torch.as_tensor(img, device="cuda")
    G, O = bf().bf_weights(g, 3, 2.0, 0.1), Graph(img.astype(np.float64), shape, 3, 2.0, 0.1)
    x0 = (g * scale).reshape(-1)
    _check(G, x0, _solution(O, x0, shift), TOL_F32, steps, may_end, shift=shift, precond=precond)


@pytest.mark.parametrize("dtype,shift,precond,steps,may_end", [
    (torch.float32, 0.5, "jacobi", 100, False), (torch.float32, 0.5, "identity", 95, True),
    (torch.float32, 0.1, "jacobi", 160, False), (torch.float32, 5.0, "jacobi", 60, True),
    (torch.float64, 0.5, "jacobi", 800, False), (torch.float64, 5.0, "jacobi", 480, True),
    (torch.float64, 0.5, "identity", 800, False), (torch.float64, 5.0, "identity", 320, True)])
def test_signals(dtype, shift, precond, steps, may_end):
    rng = np.random.default_rng(1)
    s = np.repeat(rng.uniform(0, 1, 103), 40)[:4096] + 0.1 * rng.standard_normal(4096)
    x0 = torch.as_tensor(s, device="cuda").to(dtype)
    G, O = bf().bf_weights(x0, 5, 3.0, 0.1), Graph(host(x0), (1, 4096), 5, 3.0, 0.1)
    tol = TOL_F64 if dtype == torch.float64 else TOL_F32
    _check(G, x0, _solution(O, x0, shift), tol, steps, may_end, shift=shift, precond=precond)


@pytest.mark.parametrize("radius,shift,precond,steps", [(1, 5.0, "jacobi", 40), (2, 5.0, "jacobi", 80),
                                                        (2, 50.0, "identity", 40), (3, 5.0, "jacobi", 80),
                                                        (3, 50.0, "identity", 40)])
def test_guided_images(radius, shift, precond, steps):
    shape = (66, 130)
    img = np.random.default_rng(1).uniform(0, 1, shape).astype(np.float32)
    g = torch.as_tensor(img, device="cuda")
    G, O = bf().guided_graph(g, radius, 0.01), GuidedGraph(img.astype(np.float64), shape, radius, 0.01)
    x0 = g.reshape(-1).clone()
    _check(G, x0, _solution(O, x0, shift), TOL_F32, steps, True, shift=shift, precond=precond)
