"""helm_gamma_solve at the edges of its passes: the smallest grids, odd and even lengths (the folded
transform's middle node), lengths around one round of threads, lines beyond the shared-memory
scratch and more vectors than a batch.  Reference: the Kronecker eigen-decomposition by numpy's
FP64 eigh of the two path-graph Laplacians.  Bound: the result's error is at most a few n eps times
the condition of the scaling, here below 1e-3 / 1e-6 x eigenvalue ratios; 1e-11 leaves two digits."""
import numpy as np
import pytest
import torch

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu


def _lap(n):
    d = np.full(n, 2.0)
    d[[0, -1]] = 1.0
    return (n - 1) ** 2 * (np.diag(d) - np.diag(np.ones(n - 1), 1) - np.diag(np.ones(n - 1), -1))


@pytest.mark.parametrize("nx,nz,ncol", [(2, 2, 1), (2, 3, 2), (3, 5, 17), (16, 17, 3), (64, 33, 1), (129, 128, 2), (255, 9, 1),
                                        (5, 520, 2), (4, 6100, 1), (6200, 3, 2)])
def test_matches_eigendecomposition(nx, nz, ncol):
    rng = np.random.default_rng(nx + nz)
    R = rng.standard_normal((ncol, nx * nz))
    alpha0, mu = 1e-3, 1e-2
    if max(nx, nz) > 1000:   # eigenvectors of the path graph in closed form (an eigh of 6200 takes minutes)
        def eig(n):
            a = np.arange(n)
            C = np.cos(np.pi * np.outer(a, 2 * a + 1) / (2 * n)) * np.sqrt(2.0 / n)
            C[0] = np.sqrt(1.0 / n)
            return (n - 1) ** 2 * (2.0 - 2.0 * np.cos(np.pi * a / n)), C.T
    else:
        def eig(n):
            return np.linalg.eigh(_lap(n))
    lx, Qx = eig(nx)
    lz, Qz = eig(nz)
    out = hm.helm_gamma_solve(nx, nz, alpha0, mu, torch.tensor(R, device="cuda")).cpu().numpy()
    for c in range(ncol):
        T = Qx.T @ R[c].reshape(nx, nz) @ Qz / (alpha0 * (lx[:, None] + lz[None, :]) + mu)
        ref = (Qx @ T @ Qz.T).reshape(-1)
        assert np.linalg.norm(out[c] - ref) <= 1e-11 * np.linalg.norm(ref)
