"""The run-blocked one-column kernels (7 x 7 window, weights on the fly) at the edges of
their tiles: degree, the L-type operators, the BF step and the CG filter against the FP64
oracle on images around the 64 x 16 tile and smaller than a run, with rows that are whole
16-byte vectors and rows that are not, operands off the 16-byte grid and in a strided block,
and an infinite range width.

Bounds: a weight is an exponential of an FP32 exponent e with relative error about
(2 + |e|) 2^-24 ln 2 e, |e| < 20 for weights above 1e-6; sums of 48 such terms, relative to
the norm of the result, stay below 5e-6 (the repository's 1e-5 bar for FP32 results)."""
import numpy as np
import pytest
import torch

from oracle import solvers
from oracle.graph import Graph
from paper_1509_02468_gb300 import synth
from tests.gpu_helpers import bf, host, rel_l2

pytestmark = pytest.mark.gpu
TOL = 5e-6
SHAPES = [(1, 1), (1, 3), (3, 2), (7, 64), (16, 63), (17, 65), (33, 68), (15, 130), (50, 192), (61, 257)]


def _image(shape, seed):
    if min(shape) < 8:
        return np.random.default_rng(seed).uniform(0.0, 1.0, shape).astype(np.float32)
    return synth.polygon_image(*shape, seed=seed, polygons=5)[1]


@pytest.mark.parametrize("sigma_r", [0.08, float("inf")])
@pytest.mark.parametrize("shape", SHAPES)
def test_degree_and_operators_at_tile_edges(shape, sigma_r):
    img = _image(shape, 11)
    G = bf().bf_weights(torch.as_tensor(img).cuda(), 3, 2.0, sigma_r)
    O = Graph(img.astype(np.float64), shape, 3, 2.0, sigma_r)
    n = img.size
    assert rel_l2(host(bf().graph_degree(G)), O.d) < TOL
    x = np.random.default_rng(3).standard_normal(n).astype(np.float32)
    ops = ["L", "NSYM", "DINV_W"] + (["NDIAGL"] if n > 1 else [])
    wide = torch.zeros(n, 3, device="cuda")
    wide[:, 1] = torch.as_tensor(x).cuda()
    off = torch.zeros(n + 1, device="cuda")
    off[1:] = torch.as_tensor(x).cuda()
    for op in ops:
        ref = O.apply(op, x.astype(np.float64))
        for X in (torch.as_tensor(x).cuda(), off[1:], wide[:, 1:2]):
            Y, dots = bf().bf_apply(G, op, X, dots=True)
            got = Y.double().cpu().numpy().reshape(-1)
            scale = max(np.linalg.norm(ref), 1e-6 * np.linalg.norm(x))
            assert np.linalg.norm(got - ref) <= TOL * scale, (op, X.stride())
            assert abs(float(dots[0]) - x.astype(np.float64) @ ref) <= 2e-5 * np.linalg.norm(x) * scale


@pytest.mark.parametrize("precond", ["jacobi", "identity"])
@pytest.mark.parametrize("shape", [(3, 5), (16, 64), (17, 65), (50, 131), (64, 256)])
def test_cg_at_tile_edges(shape, precond):
    img = _image(shape, 12)
    gd = torch.as_tensor(img).cuda()
    G = bf().bf_weights(gd, 3, 2.0, 0.08)
    O = Graph(img.astype(np.float64), shape, 3, 2.0, 0.08)
    for shift in (0.0, 0.05):
        x, info, _ = bf().cg_filter(G, gd.reshape(-1), 8, precond=precond, shift=shift)
        ref = solvers.cg(O, img.astype(np.float64).reshape(-1), 8, precond=precond, shift=shift)
        assert info.iters == ref["iters"]
        assert rel_l2(host(x), ref["x"]) < 1e-5


def test_reguided_steps_on_a_ragged_image():
    img = _image((45, 67), 13)
    gd = torch.as_tensor(img).cuda()
    G = bf().bf_weights(gd, 3, 2.0, 0.08)
    x = bf().reguided_filter(G, gd.reshape(-1), 3)
    ref = solvers.reguided_iteration(img.astype(np.float64), img.shape, 3, 2.0, 0.08, 3)
    assert rel_l2(host(x), ref) < 1e-5
