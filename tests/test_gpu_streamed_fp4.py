"""Streamed references in the FP4 forms on both sides of the query count from
which blocks go through an FP4 operand (128 / 129), with ragged and one-row
blocks, loci that fill neither a word nor a 256-locus stage, and rows strided
in host memory: top-k lists and hits equal the oracle's."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher, words64  # noqa: E402


@pytest.mark.parametrize("form", [B.FORM_AUTO, B.FORM_TENSOR_FP4])
@pytest.mark.parametrize("n_q,n_refs,n_loci,block,extra", [(128, 2000, 300, 700, 0), (129, 2000, 300, 700, 3),
                                                          (130, 1025, 257, 256, 0), (300, 40, 64, 1, 1),
                                                          (260, 5000, 1000, 100_000, 0)])
def test_streamed_fp4_blocks(form, n_q, n_refs, n_loci, block, extra):
    import __graft_entry__
    __graft_entry__.build()
    rng = np.random.default_rng(n_q + n_refs)
    R = (rng.random((n_refs, n_loci)) < 0.4).astype(np.uint8)
    Q = (rng.random((n_q, n_loci)) < 0.4).astype(np.uint8)
    Q[::7] = R[rng.integers(0, n_refs, len(Q[::7]))]
    modes = (rng.random(n_q) < 0.5).astype(np.uint8)
    s = Searcher(0, form)
    w = words64(n_loci)
    refs = torch.zeros((n_refs, w + extra), dtype=torch.int64).pin_memory()
    refs[:, :w] = torch.from_numpy(oracle.pack(R).view(np.int64))
    q = torch.from_numpy(oracle.pack(Q).view(np.int64)).cuda()
    m = torch.from_numpy(modes).cuda()
    exp = oracle.select(*oracle.scores(R, Q), modes)
    sc, ix = s.topk_streamed(refs[:, :w], n_loci, q, m, 20, block_refs=block, flags=0)
    es, ei = oracle.topk(exp, 20)
    assert B.fastid_sync_status(s.ctx) == B.OK
    assert np.array_equal(sc.cpu().numpy().view(np.uint32), es) and np.array_equal(ix.cpu().numpy(), ei)
    T = int(np.percentile(exp, 3))
    oq, orr, osc = oracle.hits(exp, T)
    hq, hr, hs, hc = s.hits_streamed(refs[:, :w], n_loci, q, m, T, oq.size + 5, block_refs=block, flags=0)
    assert B.fastid_sync_status(s.ctx) == B.OK
    n = int(hc.item())
    assert n == oq.size
    assert np.array_equal(hq[:n].cpu().numpy(), oq) and np.array_equal(hr[:n].cpu().numpy(), orr)
    assert np.array_equal(hs[:n].cpu().numpy().view(np.uint32), osc)
    s.ctx.close()
