"""The persistent solve kernel of the block-cyclic-reduction factor at the edges of its tiles:
the smallest grids, line lengths around the 8-row, 32-column and 128-row steps, right-hand-side
counts around the 16 / 32 / 64 tile widths, uneven numbers of lines, against the oracle's sparse
LU.  The refinement is asked for 1e-12, so the error is at most about 40 times that on these
media; 1e-8 is the mixed path's bar.  Columns of very different magnitude share a call (the
scales are per column and line), and a zero column stays zero."""
import numpy as np
import pytest
import torch

from oracle import helmholtz as H

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,n_omega,nrhs", [
    (4, 16, 1, 1), (5, 18, 2, 17), (6, 30, 1, 16), (7, 32, 1, 32), (9, 34, 3, 33), (16, 126, 1, 64), (17, 128, 1, 65),
    (8, 130, 2, 5), (12, 256, 1, 31), (11, 258, 1, 3), (5, 514, 1, 2), (64, 20, 2, 130)])
def test_edges_match_oracle(nx, nz, n_omega, nrhs):
    rng = np.random.default_rng(1000 * nx + nz)
    c = 1.0 + 0.5 * rng.uniform(0, 1, (nx, nz))
    m = (1.0 / c ** 2).reshape(-1)
    lx = (nx - 1) / (nz - 1)
    om = np.sort(rng.uniform(2.0, 8.0, n_omega))
    B = rng.standard_normal((n_omega, nrhs, nx * nz)) + 1j * rng.standard_normal((n_omega, nrhs, nx * nz))
    B *= 10.0 ** rng.uniform(-12, 12, (n_omega, nrhs, 1))
    if nrhs > 2:
        B[:, 1] = 0.0
    op = hm.helm_assemble(nx, nz, lx, 1.0, torch.tensor(m, device="cuda"), om)
    f = hm.helm_factor(op, hm.HELM_MIXED, method=hm.HELM_FACTOR_BCR)
    Bd = torch.tensor(B, device="cuda")
    g = H.Grid(nx, nz, lx, 1.0)
    for solve, adjoint in ((hm.helm_solve, False), (hm.helm_adjoint_solve, True)):
        X = solve(f, Bd, rtol=1e-12, max_iter=20)[0].cpu().numpy()
        for q, w in enumerate(om):
            fo = H.Factor(H.helmholtz_matrix(g, m, w))
            ref = fo.adjoint_solve(B[q]) if adjoint else fo.solve(B[q])
            scale = np.linalg.norm(ref, axis=1)
            err = np.linalg.norm(X[q] - ref, axis=1)
            assert np.all(err[scale == 0] == 0.0)
            assert np.max(err[scale > 0] / scale[scale > 0]) <= 1e-8


def test_the_wait_limit_gives_etimeout_and_the_next_call_is_clean():
    nx, nz = 24, 64
    rng = np.random.default_rng(3)
    m = (1.0 / (1.0 + 0.5 * rng.uniform(0, 1, (nx, nz))) ** 2).reshape(-1)
    op = hm.helm_assemble(nx, nz, 1.0, 1.0, torch.tensor(m, device="cuda"), [5.0, 7.0])
    f = hm.helm_factor(op, hm.HELM_MIXED, method=hm.HELM_FACTOR_BCR)
    B = torch.tensor(rng.standard_normal((2, 9, nx * nz)) + 0j, device="cuda")
    ref, _ = hm.helm_solve(f, B, rtol=1e-12, max_iter=20)
    try:
        hm.helm_set_wait_tries(0)
        with pytest.raises(hm.HelmError) as e:
            hm.helm_solve(f, B, rtol=1e-12, max_iter=20)
        assert e.value.status == 6   # HELM_ETIMEOUT
    finally:
        hm.helm_set_wait_tries(-1)
    X, _ = hm.helm_solve(f, B, rtol=1e-12, max_iter=20)
    assert float((X - ref).abs().max() / ref.abs().max()) <= 1e-10
