"""The CG workspace of images beyond the chip whose rows are padded (a width that is no multiple
of four): its size does not depend on the options of a call, so captured runs stay valid, and
a graph whose larger workspace cannot be had runs with the smaller one."""
import numpy as np
import pytest
import torch

from oracle import convnet as cn
from tests.gpu_helpers import TOL_F32, bf, host, rel_l2

pytestmark = pytest.mark.gpu


def _image(ny, nx):
    rng = torch.Generator(device="cuda").manual_seed(nx)
    return torch.cumsum((torch.rand((ny, nx), device="cuda", generator=rng) - 0.5) * 0.06, dim=1)


def _captured(G, x0, out, **kw):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        bf().cg_filter(G, x0, 4, out=out, sync=False, **kw)
    return graph


def _net():
    return bf().Net([np.asarray(w, np.float32) for w in cn.jacobi_weights()])


def test_capture_after_a_call_with_another_preconditioner():
    g = _image(1103, 1201)
    G, x0 = bf().bf_weights(g, 3, 2.0, 0.08), g.reshape(-1)
    bf().cg_filter(G, x0, 2, precond="net", net=_net())          # sizes the workspace
    out = torch.empty_like(x0)
    _captured(G, x0, out).replay()
    assert torch.equal(out, bf().cg_filter(G, x0, 4)[0])


def test_captured_run_survives_a_call_with_another_preconditioner():
    g = _image(1103, 1201)
    G, x0, net = bf().bf_weights(g, 3, 2.0, 0.08), g.reshape(-1), _net()
    ref = bf().cg_filter(G, x0, 4, precond="net", net=net)[0]
    out = torch.empty_like(x0)
    graph = _captured(G, x0, out, precond="net", net=net)
    bf().cg_filter(G, x0, 4)
    out.zero_()
    graph.replay()
    assert rel_l2(host(out), host(ref)) < TOL_F32


def test_smaller_workspace_where_the_larger_cannot_be_had():
    ny, nx = 8661, 8663                                          # 0.3 GB per vector
    g = _image(ny, nx)
    x0, out = g.reshape(-1), torch.empty(ny * nx, device="cuda")
    G = bf().bf_weights(g, 3, 2.0, 0.08)
    ref = bf().cg_filter(G, x0, 3)[0]
    H = bf().bf_weights(g, 3, 2.0, 0.08)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = 6 * 4 * ny * nx + (64 << 20)                          # between five and eight vectors
    filler = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        info = bf().cg_filter(H, x0, 3, out=out)[1]
    finally:
        del filler
        torch.cuda.empty_cache()
    assert info.iters == 3
    assert ((out - ref).norm() / ref.norm()).item() < TOL_F32
    again = bf().cg_filter(H, x0, 3)[0]                          # stays with it: same run
    assert torch.equal(out, again)
