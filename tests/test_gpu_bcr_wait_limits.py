"""The block-cyclic-reduction solve and factor with short wait limits: the waits give up somewhere on the
way, the call says so within the drain's time, and the next one is clean."""
import time

import numpy as np
import pytest
import torch

hm = pytest.importorskip("paper_2301_10762_gb300.helm")

pytestmark = pytest.mark.gpu

ETIMEOUT = 6


@pytest.mark.parametrize("tries", [1, 8, 64, 512])
def test_short_wait_limits(tries):
    nx, nz = 40, 160
    rng = np.random.default_rng(3)
    m = (1.0 / (1.0 + 0.5 * rng.uniform(0, 1, (nx, nz))) ** 2).reshape(-1)
    op = hm.helm_assemble(nx, nz, 1.0, 1.0, torch.tensor(m, device="cuda"), [5.0, 7.0])
    f = hm.helm_factor(op, hm.HELM_MIXED, method=hm.HELM_FACTOR_BCR)
    B = torch.tensor(rng.standard_normal((2, 33, nx * nz)) + 0j, device="cuda")
    ref, _ = hm.helm_solve(f, B, rtol=1e-12, max_iter=20)
    try:
        hm.helm_set_wait_tries(tries)
        for call in (lambda: hm.helm_solve(f, B, rtol=1e-12, max_iter=20),
                     lambda: hm.helm_factor(op, hm.HELM_MIXED, method=hm.HELM_FACTOR_BCR).close()):
            t = time.perf_counter()
            try:
                call()
            except hm.HelmError as e:
                assert e.status == ETIMEOUT
            assert time.perf_counter() - t < 5.0
    finally:
        hm.helm_set_wait_tries(-1)
    X, _ = hm.helm_solve(f, B, rtol=1e-12, max_iter=20)
    assert float((X - ref).abs().max() / ref.abs().max()) <= 1e-10
