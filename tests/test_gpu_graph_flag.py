"""A refused guide leaves nothing behind: the graph's non-finite flag is cleared before the call
that refused it returns, whatever else is queued on its stream, so the next call on another
stream is judged by its own guide."""
import threading
import time

import numpy as np
import pytest
import torch

from oracle.graph import Graph
from tests.gpu_helpers import bf, host

pytestmark = pytest.mark.gpu

SECOND = 2_000_000_000                       # cycles of torch.cuda._sleep, about


@pytest.mark.parametrize("kind", ["onthefly", "stored_f32", "guided"])
def test_next_call_on_another_stream(kind):
    img = np.random.default_rng(3).uniform(0, 1, (40, 72)).astype(np.float32)
    good = torch.as_tensor(img, device="cuda")
    bad = good.clone()
    bad[7, 9] = float("nan")
    G = (bf().guided_graph(good, 2, 0.01) if kind == "guided"
         else bf().bf_weights(good, 3, 2.0, 0.1, weight_mode=kind))
    d0 = bf().graph_degree(G)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()

    def more():                              # queued while the refusing call waits for its kernel
        time.sleep(0.1)
        with torch.cuda.stream(a):
            torch.cuda._sleep(SECOND)

    with torch.cuda.stream(a):
        torch.cuda._sleep(SECOND // 2)
    t = threading.Thread(target=more)
    t.start()
    with pytest.raises(bf().BFError) as ei:
        bf().graph_update(G, bad, stream=a)
    assert ei.value.code == bf().BF_ENONFINITE
    bf().graph_update(G, good, stream=b)     # not refused by what is left of the call before
    t.join()
    torch.cuda.synchronize()
    assert torch.equal(bf().graph_degree(G), d0)
    with pytest.raises(bf().BFError):
        bf().graph_update(G, bad, stream=b)
    bf().graph_update(G, good, stream=a)
    if kind == "onthefly":
        O = Graph(img.astype(np.float64), img.shape, 3, 2.0, 0.1)
        np.testing.assert_allclose(host(bf().graph_degree(G)), O.d, rtol=1e-5)
