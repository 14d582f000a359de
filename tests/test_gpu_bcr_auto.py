"""The automatic choice of block cyclic reduction on lines of 96 to 191 nodes and on odd lines (which
get a decoupled node): taken on sizes (at least 96 lines, blocks within 16 GB), and taken back where an eliminated block is nearly
singular: a slow disc of m = 36 in m = 1 on 96 x 96 has a mode trapped between the lines 32 and 64 at w
= 5.548174513413695, and the inverse of the block of line 48 an entry of 5e3 (the limit is 2^9 / 4).
|A^{-1}| |b| / |x| of the medium itself is below 1e2 for random b there and at w = 5, so a residual of
1e-12 leaves an error below 1e-10; 1e-8 is the mixed path's bar."""
import numpy as np
import pytest
import torch

from oracle import helmholtz as H

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu

AUTO = [(96, 96, 1, "bcr"), (130, 98, 2, "bcr"), (97, 190, 1, "bcr"), (95, 96, 1, "line"), (96, 94, 1, "line"),
        (96, 97, 1, "bcr"), (97, 193, 1, "bcr"), (96, 95, 1, "line"), (95, 193, 1, "line"), (40, 190, 1, "line"), (96, 96, 406, "line")]


@pytest.mark.parametrize("nx,nz,n_omega,want", AUTO)
def test_automatic_choice_on_sizes(nx, nz, n_omega, want):
    m = np.full(nx * nz, 0.25)
    op = hm.helm_assemble(nx, nz, 1.0, 1.0, torch.tensor(m, device="cuda"), np.linspace(5.0, 9.0, n_omega))
    f = hm.helm_factor(op, hm.HELM_MIXED)
    assert f.method == (hm.HELM_FACTOR_BCR if want == "bcr" else hm.HELM_FACTOR_LINE)


@pytest.mark.parametrize("w,want", [(5.548174513413695, "line"), (5.0, "bcr")])
def test_a_trapped_mode_takes_the_line_factor(w, want):
    n = 96
    x = np.linspace(0.0, 1.0, n)
    X, Z = np.meshgrid(x, x, indexing="ij")
    m = np.where((X - 48 / 95) ** 2 + (Z - 0.5) ** 2 < 0.25 ** 2, 36.0, 1.0).reshape(-1)
    op = hm.helm_assemble(n, n, 1.0, 1.0, torch.tensor(m, device="cuda"), [w])
    f = hm.helm_factor(op, hm.HELM_MIXED)
    assert f.method == (hm.HELM_FACTOR_BCR if want == "bcr" else hm.HELM_FACTOR_LINE)
    rng = np.random.default_rng(11)
    B = rng.standard_normal((1, 5, n * n)) + 1j * rng.standard_normal((1, 5, n * n))
    Y = hm.helm_solve(f, torch.tensor(B, device="cuda"), rtol=1e-12, max_iter=20)[0].cpu().numpy()
    ref = H.Factor(H.helmholtz_matrix(H.Grid(n, n, 1.0, 1.0), m, w)).solve(B[0])
    assert np.max(np.linalg.norm(Y[0] - ref, axis=1) / np.linalg.norm(ref, axis=1)) <= 1e-8


@pytest.mark.parametrize("nx,nz,n_omega,nrhs", [(96, 97, 2, 17), (97, 127, 1, 1), (100, 129, 1, 65), (99, 159, 1, 3),
                                                (96, 257, 1, 5)])
def test_odd_lines_match_oracle(nx, nz, n_omega, nrhs):
    """Residuals of 1e-12 (FP32 pairs) and 1e-13 (then FP64), below 1e-10 of error with |A^{-1}| |b| / |x|
    below 1e2 on these media; 1e-8 is the mixed path's bar.  A factor's first call and one with more
    columns, the working-array solve, and the adjoint."""
    rng = np.random.default_rng(100 * nx + nz)
    m = (1.0 / (1.0 + 0.5 * rng.uniform(0, 1, (nx, nz))) ** 2).reshape(-1)
    om = np.sort(rng.uniform(4.0, 9.0, n_omega))
    op = hm.helm_assemble(nx, nz, 1.0, 1.0, torch.tensor(m, device="cuda"), om)
    f = hm.helm_factor(op, hm.HELM_MIXED)
    assert f.method == hm.HELM_FACTOR_BCR
    B = rng.standard_normal((n_omega, nrhs, nx * nz)) + 1j * rng.standard_normal((n_omega, nrhs, nx * nz))
    Bd = torch.tensor(B, device="cuda")
    fo = [H.Factor(H.helmholtz_matrix(H.Grid(nx, nz, 1.0, 1.0), m, w)) for w in om]
    first = Bd[:, :1].contiguous()
    runs = [(hm.helm_solve(f, first, rtol=1e-12, max_iter=20)[0], "solve", 1),
            (hm.helm_solve(f, Bd, rtol=1e-13, max_iter=20)[0], "solve", nrhs),
            (hm.helm_adjoint_solve(f, Bd, rtol=1e-12, max_iter=20)[0], "adjoint_solve", nrhs),
            (torch.empty_like(first), "solve", 1)]
    hm.helm_solve_noalloc(f, first, runs[3][0], rtol=1e-12, max_iter=20)
    for X, how, n in runs:
        X = X.cpu().numpy()
        for q in range(n_omega):
            ref = getattr(fo[q], how)(B[q, :n])
            assert np.max(np.linalg.norm(X[q] - ref, axis=1) / np.linalg.norm(ref, axis=1)) <= 1e-8


def test_a_solve_that_does_not_converge_is_repeated_with_the_line_factor():
    """One sweep leaves 1e-5 with either factor: HELM_ENOCONV as ever, but an automatic factor has become
    the line factor by then, and the next call uses it; an explicit one stays."""
    nx, nz = 97, 99
    rng = np.random.default_rng(7)
    m = (1.0 / (1.0 + 0.5 * rng.uniform(0, 1, (nx, nz))) ** 2).reshape(-1)
    op = hm.helm_assemble(nx, nz, 1.0, 1.0, torch.tensor(m, device="cuda"), [6.0])
    B = rng.standard_normal((1, 4, nx * nz)) + 1j * rng.standard_normal((1, 4, nx * nz))
    Bd = torch.tensor(B, device="cuda")
    f = hm.helm_factor(op, hm.HELM_MIXED)
    assert f.method == hm.HELM_FACTOR_BCR
    with pytest.raises(hm.HelmError):
        hm.helm_solve(f, Bd, rtol=1e-12, max_iter=1)
    assert f.method == hm.HELM_FACTOR_LINE
    Y = hm.helm_solve(f, Bd, rtol=1e-12, max_iter=20)[0].cpu().numpy()
    ref = H.Factor(H.helmholtz_matrix(H.Grid(nx, nz, 1.0, 1.0), m, 6.0)).solve(B[0])
    assert np.max(np.linalg.norm(Y[0] - ref, axis=1) / np.linalg.norm(ref, axis=1)) <= 1e-8
    m2 = np.full(24 * 32, 0.5)
    op2 = hm.helm_assemble(24, 32, 1.0, 1.0, torch.tensor(m2, device="cuda"), [6.0])
    f2 = hm.helm_factor(op2, hm.HELM_MIXED, method=hm.HELM_FACTOR_BCR)
    B2 = torch.tensor(rng.standard_normal((1, 2, 24 * 32)) + 0j, device="cuda")
    with pytest.raises(hm.HelmError):
        hm.helm_solve(f2, B2, rtol=1e-12, max_iter=1)
    assert f2.method == hm.HELM_FACTOR_BCR
