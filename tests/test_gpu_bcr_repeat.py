"""What an unconverged solve leaves of an automatic block-cyclic-reduction factor: a limit that no factor
meets (one sweep, an rtol below FP64's floor, a right-hand side that is not finite) does not cost it.
References by the oracle at the mixed path's bar."""
import numpy as np
import pytest
import torch

from oracle import helmholtz as H

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu

NX, NZ, W = 97, 99, 6.0


def _setup():
    rng = np.random.default_rng(17)
    m = (1.0 / (1.0 + 0.5 * rng.uniform(0, 1, (NX, NZ))) ** 2).reshape(-1)
    op = hm.helm_assemble(NX, NZ, 1.0, 1.0, torch.tensor(m, device="cuda"), [W])
    f = hm.helm_factor(op, hm.HELM_MIXED)
    assert f.method == hm.HELM_FACTOR_BCR
    B = rng.standard_normal((1, 4, NX * NZ)) + 1j * rng.standard_normal((1, 4, NX * NZ))
    return op, f, B, H.Factor(H.helmholtz_matrix(H.Grid(NX, NZ, 1.0, 1.0), m, W)).solve(B[0])


def _check(X, ref):
    assert np.max(np.linalg.norm(X.cpu().numpy()[0] - ref, axis=1) / np.linalg.norm(ref, axis=1)) <= 1e-8


@pytest.mark.parametrize("how", ["solve", "noalloc"])
def test_a_sweep_limit_does_not_cost_the_factor(how):
    op, f, B, ref = _setup()
    Bd = torch.tensor(B, device="cuda")
    with pytest.raises(hm.HelmError):
        hm.helm_solve(f, Bd, rtol=1e-12, max_iter=1)
    X = torch.empty_like(Bd)
    if how == "solve":
        hm.helm_solve(f, Bd, X, rtol=1e-12, max_iter=20)
    else:
        Y = torch.empty_like(Bd[:, :2].contiguous())
        hm.helm_solve_noalloc(f, Bd[:, :2].contiguous(), Y, rtol=1e-12, max_iter=20)
        _check(Y, ref[:2])
        hm.helm_solve(f, Bd, X, rtol=1e-12, max_iter=20)
    assert f.method == hm.HELM_FACTOR_BCR
    _check(X, ref)
    with pytest.raises(hm.HelmError):   # once per factor
        hm.helm_solve(f, Bd, rtol=1e-12, max_iter=1)
    assert f.method == hm.HELM_FACTOR_BCR


@pytest.mark.parametrize("limit", ["rtol", "nan"])
def test_no_repeat_where_no_factor_converges(limit):
    op, f, B, ref = _setup()
    Bd = torch.tensor(B, device="cuda")
    bad = Bd.clone()
    if limit == "nan":
        bad[0, 0, 0] = float("nan")
    X = torch.zeros_like(Bd)
    with pytest.raises(hm.HelmError):
        hm.helm_solve(f, bad, X, rtol=0.0 if limit == "rtol" else 1e-10, max_iter=4)
    assert f.method == hm.HELM_FACTOR_BCR
    if limit == "rtol":   # four sweeps are at the floor
        _check(X, ref)
    hm.helm_solve(f, Bd, X, rtol=1e-12, max_iter=20)
    _check(X, ref)
