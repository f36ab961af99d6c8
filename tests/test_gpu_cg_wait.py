"""The one-launch CG's bounded waits: with a CTA that never sends anything every other one gives
up (1 s), the call reports BF_ETIMEOUT, x_out holds what the others had, and the next run on
the same graph is right."""
import numpy as np
import pytest
import torch

from paper_1509_02468_gb300 import synth
from tests.gpu_helpers import bf

pytestmark = pytest.mark.gpu


def _graph(kind):
    if kind.startswith("signal"):
        x = torch.as_tensor(np.random.default_rng(2).uniform(0, 1, 4096), device="cuda")
        x = x if kind == "signal_f64" else x.float()
        return bf().bf_weights(x, 5, 3.0, 0.1), x
    g = torch.as_tensor(synth.polygon_image(130, 203, 5, polygons=6)[1], device="cuda").float()
    G = bf().guided_graph(g, 2, 0.01) if kind == "guided" else bf().bf_weights(g, 3, 2.0, 0.1)
    return G, g.reshape(-1).clone()


@pytest.mark.parametrize("kind,absent", [("signal_f64", 0), ("signal_f32", 1), ("image", 0), ("image", 1), ("guided", 0)])
def test_wait_gives_up(kind, absent):
    G, x0 = _graph(kind)
    ref, info, _ = bf().cg_filter(G, x0, 6)
    out = torch.full_like(x0, -3.0)
    with pytest.raises(bf().BFError) as ei:
        bf().cg_wait_test(G, x0, 6, absent, out=out)
    assert ei.value.code == bf().BF_ETIMEOUT
    written = out != -3.0
    assert written.any() and not written.all()               # all parts but the absent one
    assert torch.equal(out[written], x0[written])
    assert written.sum().item() >= x0.numel() // 2
    x, again, _ = bf().cg_filter(G, x0, 6)
    assert torch.equal(x, ref) and again.iters == info.iters == 6


def test_other_forms_are_refused():
    g = torch.rand(64, 64, device="cuda")
    G = bf().bf_weights(g, 2, 2.0, 0.1)
    with pytest.raises(bf().BFError) as ei:
        bf().cg_wait_test(G, g.reshape(-1))
    assert ei.value.code == bf().BF_EINVAL
