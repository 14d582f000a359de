"""helm_gamma_solve with more vectors than its scratch takes at a time (64 MB: sixteen up to 724^2, one on
long lines, whose vectors are in global memory), lengths of more than a line per SM, and few long lines,
which several CTAs share.  Reference and
bound as tests/test_gpu_gamma_edges.py: the eigenvectors of the path graphs in closed form, 1e-11."""
import numpy as np
import pytest
import torch

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu


def _eig(n):
    a = np.arange(n)
    C = np.cos(np.pi * (np.outer(a, 2 * a + 1) % (4 * n)) / (2 * n)) * np.sqrt(2.0 / n)
    C[0] = np.sqrt(1.0 / n)
    return (n - 1) ** 2 * (2.0 - 2.0 * np.cos(np.pi * a / n)), C


@pytest.mark.parametrize("nx,nz,ncol", [(153, 160, 2), (305, 224, 1), (800, 730, 18), (6100, 300, 3), (40, 6050, 4), (3000, 500, 2),
                                        (30, 2000, 2), (1000, 40, 1), (64, 257, 3), (129, 2, 1), (3, 259, 20), (6300, 5, 17)])
def test_matches_eigendecomposition(nx, nz, ncol):
    rng = np.random.default_rng(nx + nz)
    R = rng.standard_normal((ncol, nx, nz))
    alpha0, mu = 1e-3, 1e-2
    (lx, Cx), (lz, Cz) = _eig(nx), _eig(nz)
    out = hm.helm_gamma_solve(nx, nz, alpha0, mu, torch.tensor(R.reshape(ncol, -1), device="cuda")).cpu().numpy()
    for c in range(ncol):
        ref = (Cx.T @ (Cx @ R[c] @ Cz.T / (alpha0 * (lx[:, None] + lz[None, :]) + mu)) @ Cz).reshape(-1)
        assert np.linalg.norm(out[c] - ref) <= 1e-11 * np.linalg.norm(ref)
