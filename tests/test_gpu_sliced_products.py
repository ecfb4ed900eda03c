"""FP64 local products on the tensor cores by exact digit slices: the block operator at the edges of the 128 x 64 output
tiles and 64-wide blocks of the product, against the oracle (FP64 operator bar of the parity tests, 1e-10)."""
import numpy as np
import pytest

from fetirp_gen import elastic_grid, heat_grid
from oracle.feti import FetiOracle

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_1208_6387_gb300.fetirp")

# (n_b, right-hand sides): an odd number of row tiles with a ragged last one; exactly full tiles in every dimension;
# an even number of row tiles and a second column tile of 17; one column tile of 16 (n_b >= 1024)
CASES = {
    "n_b 294, R 216": lambda: elastic_grid(4, (3, 3, 3), k=8, seed=2),
    "n_b 256, R 256": lambda: heat_grid(64, (8, 8), k=4, seed=3),
    "n_b 456, R 81": lambda: elastic_grid(5, (3, 3, 3), k=3, seed=4),
    "n_b 1158, R 16": lambda: elastic_grid(8, (2, 2, 1), k=4, seed=5),
}


def _context(prob):
    assert prob.patterns[0].n_b ** 2 * prob.n_occ * prob.k >= 1 << 24   # large enough for the sliced product
    ctx = F.fetirp_create(F.fetirp_default_options())
    F.load_problem(ctx, prob)
    F.fetirp_prepare(ctx, prob.n_lambda, prob.c)
    return ctx


@pytest.mark.parametrize("name", list(CASES))
def test_sliced_apply_matches_oracle(name):
    prob = CASES[name]()
    V = np.random.default_rng(0).standard_normal((prob.n_lambda, prob.k))
    ctx = _context(prob)
    try:
        Q = F.fetirp_apply_block(ctx, V)
        # scaling a column by a power of two scales every FP64 operation exactly, and the slices move with the exponent
        scale = 2.0 ** np.linspace(-300, 300, prob.k).round()
        assert np.array_equal(F.fetirp_apply_block(ctx, V * scale), Q * scale)
        # a column of zeros gives zeros; a NaN spoils its own column only
        W = V.copy()
        W[:, 0] = 0.0
        W[3, 1] = np.nan
        R = F.fetirp_apply_block(ctx, W)
        assert not R[:, 0].any() and np.isnan(R[:, 1]).all() and np.array_equal(R[:, 2:], Q[:, 2:])
    finally:
        F.fetirp_destroy(ctx)
    ref = FetiOracle(prob).PtFP(V)
    assert np.linalg.norm(Q - ref) <= 1e-10 * np.linalg.norm(ref)
