"""Device memory of the sliced FP64 products: a pattern's digit slices (16 bytes per entry of S^+) come with the first product
that takes them and not with the factorisation; without memory for them, and under a stream capture that comes first, the
products run as FP64 FMAs."""
import numpy as np
import pytest

from fetirp_gen import elastic_grid
from oracle.feti import FetiOracle

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_1208_6387_gb300.fetirp")


class Allocator:
    """Hooks on cudaMalloc'd torch memory that count what is out and can refuse everything from a size on."""

    def __init__(self):
        import torch
        self.torch, self.out, self.limit = torch, {}, None
        self.hooks = dict(alloc=F.ALLOC_FN(self._alloc), free=F.FREE_FN(self._free))

    def _alloc(self, nbytes, stream, user):
        if self.limit is not None and nbytes >= self.limit:
            return None
        ptr = self.torch.cuda.caching_allocator_alloc(int(nbytes), device=0, stream=int(stream or 0))
        self.out[ptr] = int(nbytes)
        return ptr

    def _free(self, ptr, user):
        del self.out[int(ptr)]
        self.torch.cuda.caching_allocator_delete(int(ptr))

    @property
    def bytes(self):
        return sum(self.out.values())


@pytest.fixture(scope="module")
def structure():
    prob = elastic_grid(5, (3, 3, 3), k=8, seed=4)   # n_b = 456, 216 right-hand sides
    V = np.random.default_rng(0).standard_normal((prob.n_lambda, prob.k))
    return prob, V, FetiOracle(prob).PtFP(V)


def _context(prob, **kw):
    ctx = F.fetirp_create(F.fetirp_default_options(**kw))
    F.load_problem(ctx, prob)
    F.fetirp_prepare(ctx, prob.n_lambda, prob.c)
    return ctx


def test_slices_come_with_the_first_product(structure):
    prob, V, ref = structure
    nb = prob.patterns[0].n_b
    mem = Allocator()
    ctx = _context(prob, **mem.hooks)
    try:
        F.fetirp_apply_block(ctx, V, F.PRECISIONS["tf32x3"])
        before = mem.bytes
        Q = F.fetirp_apply_block(ctx, V)
        assert mem.bytes - before >= 16 * nb * nb
        held = mem.bytes
        F.fetirp_factorize(ctx)                      # the slices follow the factorisation in the memory they have
        F.fetirp_prepare(ctx, prob.n_lambda, prob.c)
        assert np.array_equal(F.fetirp_apply_block(ctx, V), Q) and mem.bytes <= held
    finally:
        F.fetirp_destroy(ctx)
    assert not mem.out
    assert np.linalg.norm(Q - ref) <= 1e-10 * np.linalg.norm(ref)


def test_narrower_products_leave_the_scratch_in_place(structure):
    """The scratch of the first sliced product, a narrow one here, is that of the whole block: what a program captured at
    any width stays valid."""
    prob, V, ref = structure
    mem = Allocator()
    ctx = _context(prob, **mem.hooks)
    try:
        F.fetirp_apply_block(ctx, np.ascontiguousarray(V[:, :3]))   # 81 right-hand sides: just above the line
        held = dict(mem.out)
        for k in (8, 5, 3):
            Q = F.fetirp_apply_block(ctx, np.ascontiguousarray(V[:, :k]))
            assert np.linalg.norm(Q - ref[:, :k]) <= 1e-10 * np.linalg.norm(ref[:, :k])
        assert mem.out == held
    finally:
        F.fetirp_destroy(ctx)


def test_without_memory_for_the_slices(structure):
    prob, V, ref = structure
    nb = prob.patterns[0].n_b
    mem = Allocator()
    ctx = _context(prob, **mem.hooks)
    try:
        mem.limit = 16 * nb * nb
        Q = F.fetirp_apply_block(ctx, V)
        mem.limit = None
        R = F.fetirp_apply_block(ctx, V)
    finally:
        F.fetirp_destroy(ctx)
    assert np.linalg.norm(Q - ref) <= 1e-10 * np.linalg.norm(ref)
    assert np.linalg.norm(R - ref) <= 1e-10 * np.linalg.norm(ref)


def test_first_product_under_capture(structure):
    import torch
    prob, V, ref = structure
    stream = torch.cuda.Stream()
    ctx = _context(prob, cuda_stream=stream.cuda_stream)
    try:
        v = torch.from_numpy(V).cuda()
        q = torch.zeros_like(v)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            F.fetirp_apply_block_device(ctx, prob.k, v.data_ptr(), q.data_ptr())
        graph.replay()
        torch.cuda.synchronize()
        Q = q.cpu().numpy()
        R = F.fetirp_apply_block(ctx, V)
    finally:
        F.fetirp_destroy(ctx)
    assert np.linalg.norm(Q - ref) <= 1e-10 * np.linalg.norm(ref)
    assert np.linalg.norm(R - ref) <= 1e-10 * np.linalg.norm(ref)
