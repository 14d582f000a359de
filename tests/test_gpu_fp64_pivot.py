"""FP64 line factors where their pivot inversion and their shapes can go wrong: 16 x 16 pivot blocks
with small and zero diagonals (the row exchanges), ragged last blocks, the slab of sixteen CTAs
(n_z from 200) and the sweep shapes around their choice, against the oracle at the FP64 bar 1e-9."""
import numpy as np
import pytest
import torch

from oracle import helmholtz as H

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,n_omega,nrhs", [(9, 17, 2, 3), (8, 47, 1, 5), (7, 48, 3, 1), (12, 65, 1, 9), (10, 130, 2, 7),
                                                (6, 200, 1, 2), (9, 241, 1, 17)])
def test_line_factor_and_sweep_match_oracle(nx, nz, n_omega, nrhs):
    rng = np.random.default_rng(nx * nz)
    hx, hz = 1.0 / (nx - 1), 1.0 / (nz - 1)
    om = 2.0 + np.arange(n_omega)
    # the model of every third interior node brings the diagonal of A at the first frequency near 0
    c = 1.0 + 0.5 * rng.uniform(0, 1, (nx, nz))
    m = 1.0 / c ** 2
    m[1:-1:3, 1:-1:3] = 2.0 * (hz / hx + hx / hz) / (om[0] ** 2 * hx * hz) * (1.0 + 1e-9 * rng.standard_normal())
    B = rng.standard_normal((n_omega, nrhs, nx * nz)) + 1j * rng.standard_normal((n_omega, nrhs, nx * nz))
    op = hm.helm_assemble(nx, nz, 1.0, 1.0, torch.tensor(m.reshape(-1), device="cuda"), om)
    f = hm.helm_factor(op, hm.HELM_FP64)
    g = H.Grid(nx, nz, 1.0, 1.0)
    Bd = torch.tensor(B, device="cuda")
    for solve, adjoint in ((hm.helm_solve, False), (hm.helm_adjoint_solve, True)):
        X = solve(f, Bd)[0].cpu().numpy()
        for q, w in enumerate(om):
            fo = H.Factor(H.helmholtz_matrix(g, m.reshape(-1), w))
            ref = fo.adjoint_solve(B[q]) if adjoint else fo.solve(B[q])
            assert np.max(np.linalg.norm(X[q] - ref, axis=1) / np.linalg.norm(ref, axis=1)) <= 1e-9
