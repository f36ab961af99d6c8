"""L X on blocks with stored weights (7 x 7 window) at the edges of the 32-pixel tiles: every
block width with a kernel of its own, rows shorter and longer than a tile, blocks with a
padded row stride, both storage types; against the exact FP64 operator of the stored weights.
The bound is the repository's 1e-5 for FP32 results."""
import numpy as np
import pytest
import torch

from oracle.graph import Graph
from tests.gpu_helpers import TOL_F32, bf, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["stored_f32", "stored_bf16"])
@pytest.mark.parametrize("shape", [(3, 5), (31, 33), (38, 38), (65, 97), (40, 128)])
def test_blocks_with_stored_weights(shape, mode):
    rng = np.random.default_rng(shape[0])
    img = rng.uniform(0, 0.3, shape).astype(np.float32)
    G = bf().bf_weights(torch.as_tensor(img, device="cuda"), 3, 2.0, 0.1, weight_mode=mode)
    O = Graph.from_taps(host(bf().graph_export_weights(G)), shape, 3)
    n = img.size
    for k in (4, 8, 12, 16, 32):
        wide = torch.as_tensor(rng.standard_normal((n, k + 4)).astype(np.float32), device="cuda")
        for X in (wide[:, :k], wide[:, :k].contiguous()):
            Y = bf().bf_apply(G, "L", X, Y=torch.empty((n, k + 8), device="cuda")[:, :k])
            assert rel_l2(host(Y), O.apply("L", host(X))) < TOL_F32, (k, X.stride())
