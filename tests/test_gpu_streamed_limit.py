"""Streamed calls whose blocks' FP4 operands are not allowed the memory they
would take: the call goes on over packed rows, with the same lists and hits,
and its context holds less memory.  The bound is met exactly on both sides."""
import numpy as np
import pytest

import oracle
from host import ctx_hooks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

N_Q, N_REFS, N_LOCI, K = 300, 140_000, 1000, 20
BLOCK = 131_072  # two operands of 67 MB; staging, packed rows and scratch come to 75


@pytest.fixture(scope="module")
def problem():
    import __graft_entry__
    __graft_entry__.build()
    rng = np.random.default_rng(5)
    R = (rng.random((N_REFS, N_LOCI)) < 0.4).astype(np.uint8)
    Q = (rng.random((N_Q, N_LOCI)) < 0.4).astype(np.uint8)
    Q[::7] = R[rng.integers(0, N_REFS, len(Q[::7]))]
    modes = (rng.random(N_Q) < 0.5).astype(np.uint8)
    return R, Q, modes, oracle.select(*oracle.scores(R, Q), modes)


@pytest.mark.parametrize("below", [None, 0, 1], ids=["own rule", "at the bound", "a byte below"])
def test_streamed_operand_limit(problem, tmp_path, below):
    R, Q, modes, exp = problem
    hooks = ctx_hooks(tmp_path)
    operands = 2 * BLOCK * hooks.hook_kbytes4(N_LOCI)
    s = Searcher(0, B.FORM_AUTO)
    hooks.hook_fp4_block_bytes(s.ctx.handle, -1 if below is None else operands - below)
    refs = torch.from_numpy(oracle.pack(R).view(np.int64)).pin_memory()
    q = torch.from_numpy(oracle.pack(Q).view(np.int64)).cuda()
    m = torch.from_numpy(modes).cuda()
    es, ei = oracle.topk(exp, K)
    for _ in range(2):  # the second call finds the pool's memory held
        sc, ix = s.topk_streamed(refs, N_LOCI, q, m, K, block_refs=BLOCK, flags=0)
        assert B.fastid_sync_status(s.ctx) == B.OK
        assert np.array_equal(sc.cpu().numpy().view(np.uint32), es) and np.array_equal(ix.cpu().numpy(), ei)
    held = B.fastid_memory_info(s.ctx)["pool_reserved_bytes"]
    assert (held >= operands) == (below != 1), (held, operands)
    T = int(np.percentile(exp, 2))
    oq, orr, osc = oracle.hits(exp, T)
    hq, hr, hs, hc = s.hits_streamed(refs, N_LOCI, q, m, T, oq.size + 5, block_refs=BLOCK, flags=0)
    assert B.fastid_sync_status(s.ctx) == B.OK
    n = int(hc.item())
    assert n == oq.size
    assert np.array_equal(hq[:n].cpu().numpy(), oq) and np.array_equal(hr[:n].cpu().numpy(), orr)
    assert np.array_equal(hs[:n].cpu().numpy().view(np.uint32), osc)
    s.ctx.close()
