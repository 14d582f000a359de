"""Line factors and sweeps at the lines where their shapes change, on few lines, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import helmholtz as H

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu


def _case(nx, nz, n_omega, nrhs):
    rng = np.random.default_rng(1000 * nx + nz)
    m = (1.0 / (1.0 + 0.5 * rng.uniform(0, 1, (nx, nz))) ** 2).reshape(-1)
    om = np.sort(rng.uniform(2.0, 8.0, n_omega))
    B = rng.standard_normal((n_omega, nrhs, nx * nz)) + 1j * rng.standard_normal((n_omega, nrhs, nx * nz))
    lx = (nx - 1) / (nz - 1)
    op = hm.helm_assemble(nx, nz, lx, 1.0, torch.tensor(m, device="cuda"), om)
    fo = [H.Factor(H.helmholtz_matrix(H.Grid(nx, nz, lx, 1.0), m, w)) for w in om]
    return op, B, np.stack([f.solve(B[q]) for q, f in enumerate(fo)])


def _error(X, ref):
    return np.max(np.linalg.norm(X.cpu().numpy() - ref, axis=2) / np.linalg.norm(ref, axis=2))


@pytest.mark.parametrize("nx,nz,method", [(5, 307, "line"), (5, 308, "line"), (6, 325, "line"), (5, 326, "line"), (5, 386, "line"), (5, 387, "line"),
                                          (6, 409, "line"), (5, 410, "line"), (7, 309, "auto"), (5, 401, "auto")])
def test_mixed_line_factor_around_the_slabs_shared_memory(nx, nz, method):
    """The complex FP32 slab of eight CTAs fits up to n_z = 307 beside the kernel's static arrays, that of
    sixteen up to 386; a limit that takes the static arrays for FP64's has 325 and 409 (odd lines on few
    lines: the automatic choice).  1e-12 asked for, 1e-8 the mixed bar."""
    op, B, ref = _case(nx, nz, 2, 3)
    f = hm.helm_factor(op, hm.HELM_MIXED, method=hm.HELM_FACTOR_LINE if method == "line" else hm.HELM_FACTOR_AUTO)
    assert f.method == hm.HELM_FACTOR_LINE
    X = hm.helm_solve(f, torch.tensor(B, device="cuda"), rtol=1e-12, max_iter=20)[0]
    assert _error(X, ref) <= 1e-8


@pytest.mark.parametrize("nx,nz,nrhs,teams", [(8, 48, 5, 2), (8, 49, 5, 2), (7, 50, 1, 2), (9, 57, 3, 2), (6, 99, 2, 2), (5, 49, 3, 1),
                                              (6, 100, 3, 1), (5, 113, 1, 1)])
def test_fp64_sweep_teams_without_idle_ctas(nx, nz, nrhs, teams, monkeypatch):
    """Line lengths that a doubled number of CTAs does not divide into filled ones (49 on 8 CTAs: seven
    rows each, the eighth none; 100 on 16: the last without rows).  FP64 bar 1e-9."""
    if teams == 1:
        monkeypatch.setenv("HELM_FACTOR_TEAMS", "1")
    op, B, ref = _case(nx, nz, 1, nrhs)
    f = hm.helm_factor(op, hm.HELM_FP64)
    assert _error(hm.helm_solve(f, torch.tensor(B, device="cuda"))[0], ref) <= 1e-9


@pytest.mark.parametrize("nx,nz,n_omega,nrhs", [(4, 4, 1, 1), (119, 10, 2, 79), (7, 5, 3, 2), (33, 31, 1, 40), (40, 33, 2, 3), (64, 64, 2, 64)])
def test_refinement_runs_on_across_short_lines(nx, nz, n_omega, nrhs):
    """The line factor's refinement takes groups of 32 nodes across lines, 2 or 8 of them a thread: columns
    that end within a group, both thread counts, the adjoint and the working-array solve.  Mixed bar 1e-8."""
    op, B, ref = _case(nx, nz, n_omega, nrhs)
    f = hm.helm_factor(op, hm.HELM_MIXED, method=hm.HELM_FACTOR_LINE)
    Bd = torch.tensor(B, device="cuda")
    assert _error(hm.helm_solve(f, Bd, rtol=1e-12, max_iter=20)[0], ref) <= 1e-8
    X = hm.helm_adjoint_solve(f, Bd.conj().resolve_conj(), rtol=1e-12, max_iter=20)[0]   # A^H conj(x) = conj(b)
    assert _error(X.conj().resolve_conj(), ref) <= 1e-8
    one = Bd[:, :1].contiguous()
    Y = torch.empty_like(one)
    hm.helm_solve_noalloc(f, one, Y, rtol=1e-12, max_iter=20)
    assert _error(Y, ref[:, :1]) <= 1e-8
