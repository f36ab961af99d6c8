"""The stored-weight block walk on images whose weight planes pass 2^31 bytes, up to the size at
which the general kernel takes over and just beyond it, against the one-column operator (64-bit
offsets) column by column.  Both sum 48 products w (x_i - x_j) <= 1 in FP32: they differ by at
most 2 x 48 x 48 x 2^-24 = 2.7e-4 per entry."""
import pytest
import torch

from tests.gpu_helpers import bf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,shape", [("stored_f32", (4701, 4703)), ("stored_f32", (4801, 5003)), ("stored_f32", (6631, 6635)),
                                        ("stored_bf16", (6631, 6635)), ("stored_f32", (6636, 6632))])
@pytest.mark.parametrize("k", [4, 8, 16])
def test_against_one_column(mode, shape, k):
    gen = torch.Generator(device="cuda").manual_seed(1)
    g = torch.rand(shape, device="cuda", generator=gen)
    G = bf().bf_weights(g, 3, 2.0, 0.5, weight_mode=mode)
    X = torch.rand((G.n, k), device="cuda", generator=gen)
    Y = bf().bf_apply(G, "L", X)
    for c in (0, k // 2, k - 1):
        y = bf().bf_apply(G, "L", X[:, c].contiguous())
        assert (Y[:, c] - y).abs().max().item() <= 2.7e-4
