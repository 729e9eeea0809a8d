"""The inner solve in one cluster per pair of right-hand sides (small lattices, few
right-hand sides) against the same solve launched step by step: lattices of 1 to 16
blocks of sites with full and partial last blocks, pairs and odd counts, a member that
has nothing to solve, and the ways a solve ends early.  The results are the same bits."""
import numpy as np
import pytest

from lattice_inputs import haar_su3_field, gaussian_spinors
from tests._gpu import lattice, to_dev, torch

pytestmark = pytest.mark.gpu

KAPPA, TOL = 0.12, 1e-10


def _solve(L, h, b, monkeypatch, stepwise, **kw):
    if stepwise:
        monkeypatch.setenv("LQCD_NO_GRAPH", "1")
    else:
        monkeypatch.delenv("LQCD_NO_GRAPH", raising=False)
    x = torch.empty_like(b)
    before = L.lqcd_launch_count()
    rc, st = L.lqcd_solve_batch(h, b, x, L.solver_params(**kw))
    return rc, st, x, L.lqcd_launch_count() - before


# 8 to 2048 sites of a parity: blocks of 128, the cluster is the next power of two
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 4, 4), (6, 4, 2, 8), (6, 6, 6, 6), (4, 4, 8, 10), (8, 8, 8, 8)])
@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("n", [1, 2, 5])
def test_cluster_solve_matches_steps(dims, prec, n, monkeypatch):
    monkeypatch.delenv("LQCD_HOP_VARIANT", raising=False)
    V = int(np.prod(dims))
    b = gaussian_spinors(dims, n, 31).reshape(n, V, 4, 3)
    if n == 5:
        b[2] = 0.0  # the first member of a pair has nothing to solve
    b = to_dev(b)
    with lattice(dims, haar_su3_field(dims, 3), KAPPA) as (L, h):
        p = L.LQCD_PREC_MIXED_FP16 if prec == "fp16" else L.LQCD_PREC_MIXED_BF16
        rc, st, x, launches = _solve(L, h, b, monkeypatch, False, tol=TOL, precision=p)
        rc2, st2, x2, launches2 = _solve(L, h, b, monkeypatch, True, tol=TOL, precision=p)
        assert rc == 0 and rc2 == 0
        assert launches < launches2 / 2  # (one launch for all inner iterations of a cycle)
        for k in range(n):
            assert st[k] == st2[k] and st[k]["status"] == 0
            assert st[k]["true_rel_residual"] <= TOL
        assert torch.equal(x, x2)  # the same terms and sums in the same order
        # the iteration cap and the wall-clock budget
        for kw, name in ((dict(tol=TOL, max_iter=3), "LQCD_ERR_NOT_CONVERGED"),
                         (dict(tol=1e-14, timeout_ms=1e-6), "LQCD_ERR_TIMEOUT")):
            rc, st, x, _ = _solve(L, h, b, monkeypatch, False, precision=p, **kw)
            rc2, st2, x2, _ = _solve(L, h, b, monkeypatch, True, precision=p, **kw)
            assert rc == rc2 == getattr(L, name)
            assert [s["status"] for s in st] == [s["status"] for s in st2]
