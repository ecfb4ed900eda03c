"""Block widths at the edges of the kernels' lane groups (4, 8, 16, 32 columns per link in G^T V, 4 columns per thread in
G A) and output tiles (right-hand sides in steps of 32), on a ragged pattern (n_b = 456): the operator and the solves
against the oracle, with the bars of the parity tests."""
import numpy as np
import pytest

from fetirp_gen import elastic_grid
from oracle.direct import direct
from oracle.feti import FetiOracle

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_1208_6387_gb300.fetirp")


@pytest.fixture(scope="module")
def structure():
    prob = elastic_grid(5, (2, 2, 2), n_patterns=2, k=8, seed=6)
    ctx = F.fetirp_create(F.fetirp_default_options())
    F.load_problem(ctx, prob)
    F.fetirp_prepare(ctx, prob.n_lambda, prob.c)
    yield prob, ctx, FetiOracle(prob)
    F.fetirp_destroy(ctx)


@pytest.mark.parametrize("k", [1, 2, 4, 5, 8, 9, 16, 17, 24, 32, 33, 64])
def test_apply_widths(structure, k):
    prob, ctx, orc = structure
    V = np.random.default_rng(k).standard_normal((prob.n_lambda, k))
    ref = orc.PtFP(V)
    for prec, tol in (("fp64", 1e-10), ("fp32", 2e-6), ("tf32x3", 1e-5), ("bf16x3", 5e-5)):
        Q = F.fetirp_apply_block(ctx, V, F.PRECISIONS[prec])
        assert np.linalg.norm(Q - ref) <= tol * np.linalg.norm(ref), prec


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8, 9, 20])
def test_solve_widths_per_phase_kernels(k):
    """The reductions of eta and W^T r for every width (FP32 products: double-single sums)."""
    prob = elastic_grid(3, (3, 3, 3), k=k, seed=7)
    us_ref, lam_ref, _, _ = direct(prob)
    ctx = F.fetirp_create(F.fetirp_default_options(precision="fp32", tol=1e-11, persistent=0))
    try:
        F.load_problem(ctx, prob)
        lam, u, _ = F.fetirp_solve(ctx, prob.n_lambda, prob.c, F.n_u(prob))
    finally:
        F.fetirp_destroy(ctx)
    assert np.linalg.norm(lam - lam_ref) <= 1e-8 * np.linalg.norm(lam_ref)
    for a, b in zip(F.split_u(prob, u), us_ref):
        assert np.linalg.norm(a - b) <= 1e-8 * np.linalg.norm(b)
