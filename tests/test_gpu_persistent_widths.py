"""The persistent iteration at the block widths that have a history update of their own (4, 8, 16 and 32 columns: row
tiles of 256, 128, 64 and 32 rows, with several history splits and a ragged last tile) and at two that do not, against
the direct solve, with the bars of the parity tests.  Device memory comes from a suballocator that hands out
256-byte blocks filled with a nonzero pattern and keeps guard bytes between them: counters and sums that start from
memory nobody cleared change the solution, and a write past a buffer's end changes its guard."""
import numpy as np
import pytest

from fetirp_gen import heat_grid
from oracle.direct import direct

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_1208_6387_gb300.fetirp")

FILL, GUARD = 0x5A, 1024


class GuardedArena:
    def __init__(self, nbytes):
        import torch
        self.arena = torch.full((nbytes,), FILL, dtype=torch.uint8, device="cuda")
        self.top = 0
        self.blocks = []
        self.hooks = F.ALLOC_FN(self._alloc), F.FREE_FN(lambda ptr, user: None)

    def _alloc(self, nbytes, stream, user):
        start = self.top
        end = start + int(nbytes)
        self.top = (end + GUARD + 255) // 256 * 256
        if self.top > self.arena.numel():
            return None   # the library reports FETIRP_ENOMEM
        self.blocks.append((end, self.top))
        return self.arena.data_ptr() + start

    def damaged(self):
        return [b for b in self.blocks if bool((self.arena[b[0]:b[1]] != FILL).any())]


@pytest.mark.parametrize("grid", [(8, 8), (7, 9)])
@pytest.mark.parametrize("k", [4, 8, 12, 16, 24, 32])
@pytest.mark.parametrize("prec", ["fp32", "auto"])
def test_persistent_widths(grid, k, prec):
    prob = heat_grid(16, grid, kappas=(1.0, 1000.0), checker=True, k=k, seed=11)
    assert persist_tiles_are_ragged(prob.n_lambda, grid)
    us_ref, lam_ref, _, _ = direct(prob)
    arena = GuardedArena(1 << 30)
    alloc, free = arena.hooks
    ctx = F.fetirp_create(F.fetirp_default_options(precision=prec, tol=5e-13, persistent=1, history_bytes=64 << 20,
                                                   alloc=alloc, free=free))
    try:
        F.load_problem(ctx, prob)
        lam, u, st = F.fetirp_solve(ctx, prob.n_lambda, prob.c, F.n_u(prob))
        assert not arena.damaged()
    finally:
        F.fetirp_destroy(ctx)
    assert st["iterations"] * k >= 128   # long enough for several splits of the history
    assert np.linalg.norm(lam - lam_ref) <= 1e-8 * np.linalg.norm(lam_ref)
    for a, b in zip(F.split_u(prob, u), us_ref):
        assert np.linalg.norm(a - b) <= 1e-8 * np.linalg.norm(b)


def persist_tiles_are_ragged(n, grid):
    """8 x 8: whole 32- and 64-row tiles, a ragged 128- and 256-row one; 7 x 9: every tile size ends in a ragged one."""
    return n % 128 != 0 and n % 256 != 0 and (grid == (8, 8) or all(n % r for r in (32, 64)))
