"""Mixed misfit gradients on grids of the block-cyclic-reduction factor (96 lines of 96 nodes and more)
against the oracle, crosswell, speeds 1.5 to 4.5.  Both solves stop at residuals of 1e-12; a residual of the
field's shape leaves up to |A^{-1}| |b| / |x| times that, some 1e3 at the lowest frequency here, and the
data residual is a tenth of the data: 1e-8, the mixed path's bar."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import helmholtz as H

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,seed", [(96, 96, 1), (150, 101, 2), (160, 160, 3), (192, 192, 4), (224, 224, 5), (224, 224, 6)])
def test_gradient_matches_oracle(nx, nz, seed):
    lx = (nx - 1) / (nz - 1)
    f = W.gaussian_random_field(nx, nz, 0.1, seed, lx=lx)
    c = 1.5 + 3.0 * (f - f.min()) / (f.max() - f.min())
    m_true = (c ** -2).reshape(nx, nz)
    m = W.gaussian_smooth(m_true, 4.0).reshape(-1)
    m_true = m_true.reshape(-1)
    om = np.array([3.0, 0.12 * min(nx, nz)])
    src = np.stack([np.full(4, 0.05 * lx), np.linspace(0.1, 0.9, 4)], 1)
    rec = np.stack([np.full(7, 0.95 * lx), np.linspace(0.08, 0.93, 7)], 1)
    g = H.Grid(nx, nz, lx, 1.0)
    data, _ = H.synthetic_data(g, m_true, om, src, rec)
    phi_o, grad_o = H.fwi_objective_gradient(g, m, om, src, rec, data, 1e-6, 1e-6)[:2]
    op = hm.helm_assemble(nx, nz, lx, 1.0, torch.tensor(m, device="cuda"), om)
    fac = hm.helm_factor(op, hm.HELM_MIXED)
    assert fac.method == hm.HELM_FACTOR_BCR
    phi, grad, _, _ = hm.fwi_misfit_grad(fac, hm.Acq(src, rec), torch.tensor(data, device="cuda"), 1e-6, 1e-6, rtol=1e-12)
    assert abs(phi - phi_o) <= 1e-8 * abs(phi_o)
    assert np.linalg.norm(grad.cpu().numpy() - grad_o) <= 1e-8 * np.linalg.norm(grad_o)
