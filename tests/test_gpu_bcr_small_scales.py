"""Small right-hand sides on grids whose cells are far from square: the blocks' entries are small there
(about 2^-17 at h_x / h_z = 1e6, against 1 on square cells) and so are the lines that they multiply,
so that the common exponent of a product's terms passes that of the smallest FP32 number.  Scaling B
by a power of two scales X, as long as the residuals (1e-12 of B) are normal numbers; 1e-8 is the mixed
path's bar."""
import numpy as np
import pytest
import torch

from oracle import helmholtz as H

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ratio", [1.0, 1e4, 1e6])
@pytest.mark.parametrize("log2b", [0, -40, -60])
def test_small_right_hand_sides(ratio, log2b):
    nx, nz, nrhs = 9, 32, 5
    rng = np.random.default_rng(5)
    lx = ratio * (nx - 1) / (nz - 1)
    m = (1.0 / (1.0 + 0.5 * rng.uniform(0, 1, (nx, nz))) ** 2).reshape(-1)
    op = hm.helm_assemble(nx, nz, lx, 1.0, torch.tensor(m, device="cuda"), [5.0])
    f = hm.helm_factor(op, hm.HELM_MIXED, method=hm.HELM_FACTOR_BCR)
    B = rng.standard_normal((1, nrhs, nx * nz)) + 1j * rng.standard_normal((1, nrhs, nx * nz))
    X = hm.helm_solve(f, torch.tensor(B * 2.0 ** log2b, device="cuda"), rtol=1e-11, max_iter=20)[0].cpu().numpy()
    ref = H.Factor(H.helmholtz_matrix(H.Grid(nx, nz, lx, 1.0), m, 5.0)).solve(B[0]) * 2.0 ** log2b
    assert np.max(np.linalg.norm(X[0] - ref, axis=1) / np.linalg.norm(ref, axis=1)) <= 1e-8
