"""helm_zinv_batched around the sizes where its kernel changes (two groups of 32 columns up to n = 64, four
above) and its 16-column steps end, for a block, a few and more than two to an SM, against numpy in 64
bits.  The blocks' condition is below 10 (a shift of 3 sqrt(n) on entries of 1): 1e-5, as for the other sizes."""
import numpy as np
import pytest
import torch

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 14, 16, 18, 32, 34, 62, 64, 66, 96, 126])
@pytest.mark.parametrize("batch", [1, 7, 321])
def test_matches_numpy_inverse(n, batch):
    rng = np.random.default_rng(n + batch)
    M = rng.standard_normal((batch, n, n)) + 1j * rng.standard_normal((batch, n, n))
    M = ((M + np.transpose(M, (0, 2, 1))) / 2 + 3.0 * np.sqrt(n) * np.eye(n)).astype(np.complex64)
    A = torch.tensor(M, device="cuda")
    ref = np.linalg.inv(M.astype(np.complex128))
    X = hm.helm_zinv_batched(A).cpu().numpy()
    assert np.max(np.linalg.norm(X - ref, axis=(1, 2)) / np.linalg.norm(ref, axis=(1, 2))) <= 1e-5
    hm.helm_zinv_batched(A, A)   # in place
    assert np.array_equal(A.cpu().numpy(), X)
