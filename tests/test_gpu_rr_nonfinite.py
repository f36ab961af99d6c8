"""Rayleigh-Ritz with entries that are not finite: status 3, and the next solve is right (the
vectors are taken by the ranks of the Ritz values, which have to be a permutation with NaNs
among them); LOBPCG on a graph without any edge weight."""
import numpy as np
import pytest
import torch

from oracle import solvers
from tests.gpu_helpers import bf, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,k", [(4, 2), (12, 4), (48, 16), (96, 32)])
def test_nonfinite_pencil(m, k):
    rng = np.random.default_rng(m)
    A = rng.standard_normal((m, m))
    A, B = A @ A.T, np.eye(m)
    for bad in (np.nan, np.inf):
        Ab = A.copy()
        Ab[m // 2, m // 2] = bad
        status = bf().rayleigh_ritz(torch.as_tensor(Ab, device="cuda"), torch.as_tensor(B, device="cuda"), k)[3]
        assert status == 3
    C, theta, _, status, _ = bf().rayleigh_ritz(torch.as_tensor(A, device="cuda"), torch.as_tensor(B, device="cuda"), k)
    assert status == 0
    np.testing.assert_allclose(host(theta), solvers.rayleigh_ritz(A, B, k)[0], atol=1e-6 * np.linalg.norm(A, 2))


def test_lobpcg_without_edges():
    """sigma_r so small that every weight underflows: L = 0, and every Ritz value is 0 or the
    run reports that its basis broke down."""
    g = torch.arange(40 * 50, device="cuda", dtype=torch.float32).view(40, 50)
    G = bf().bf_weights(g, 3, 2.0, 1e-3)
    X = torch.randn((2000, 8), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    for kmax in (1, 3):
        try:
            out = bf().lobpcg_filter(G, X, kmax)
        except bf().BFError as e:
            assert e.code in (bf().BF_EBREAKDOWN, bf().BF_ENONFINITE)
            continue
        assert out["theta"].abs().max().item() == 0.0 and torch.isfinite(out["y"]).all()
