"""Factorisation of patterns with pinned interior planes (identity rows and columns, as a caller fixes dofs): tile columns
of the factor without a tile below the diagonal, met while trailing updates are on the side stream.  S^+ against the
dense Schur complement (FP64 operator bar of the parity tests, 1e-10), and the same bits at every factorisation."""
import numpy as np
import pytest
import scipy.sparse as sp

from fetirp_gen.mesh import elastic_pattern

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_1208_6387_gb300.fetirp")


@pytest.mark.parametrize("planes", [1, 2])
def test_pinned_interior_planes(planes):
    pat = elastic_pattern(8)
    interior = np.setdiff1d(np.arange(pat.n_nodes), pat.bnd_nodes)
    nodes = interior[-planes * 7 * 7:]   # interior dofs 7^3 nodes: the last planes, after which only the boundary follows
    pinned = (3 * nodes[:, None] + np.arange(3)).ravel()
    K = pat.K.toarray()
    K[pinned, :] = 0.0
    K[:, pinned] = 0.0
    K[pinned, pinned] = 1.0
    b = (3 * pat.bnd_nodes[:, None].astype(int) + np.arange(3)).ravel()
    i = np.setdiff1d(np.arange(pat.n_dofs), b)
    schur = K[np.ix_(b, b)] - K[np.ix_(b, i)] @ np.linalg.solve(K[np.ix_(i, i)], K[np.ix_(i, b)])
    ref = np.linalg.inv(schur)
    csr = sp.csr_matrix(K)   # no stored entry couples a pinned dof
    ctx = F.fetirp_create(F.fetirp_default_options())
    try:
        pid = F.fetirp_create_pattern(ctx, pat.n_nodes, 3, csr.indptr, csr.indices, csr.data, pat.bnd_nodes, 0)
        first = F.fetirp_get_pattern(ctx, pid)[2]
        for _ in range(3):
            F.fetirp_factorize(ctx)
            assert np.array_equal(F.fetirp_get_pattern(ctx, pid)[2], first)
    finally:
        F.fetirp_destroy(ctx)
    assert np.linalg.norm(first - ref) <= 1e-10 * np.linalg.norm(ref)
