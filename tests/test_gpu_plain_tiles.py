"""The plain form's query tiles (128, 64, 32, 16): query counts on both sides
of every step of the choice, several tiles of each height, ragged references
and loci, in top-k, hit lists, both matrix widths and the allocation-free
call.  Exact integers against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

N_Q = [1, 15, 16, 17, 31, 32, 33, 47, 48, 49, 64, 65, 80, 97, 112, 128, 129, 144, 192, 193, 300, 1023, 1024, 1025]


@pytest.mark.parametrize("n_q", N_Q)
def test_plain_tiles(n_q):
    import __graft_entry__
    __graft_entry__.build()
    rng = np.random.default_rng(n_q)
    n_refs, n_loci, k = int(rng.integers(100, 3000)), int(rng.integers(1, 700)), int(rng.integers(1, 33))
    R = (rng.random((n_refs, n_loci)) < 0.4).astype(np.uint8)
    Q = (rng.random((n_q, n_loci)) < 0.4).astype(np.uint8)
    Q[::5] = R[rng.integers(0, n_refs, len(Q[::5]))]
    modes = (rng.random(n_q) < 0.5).astype(np.uint8)
    exp = oracle.select(*oracle.scores(R, Q), modes)
    s = Searcher(0, B.FORM_PLAIN)
    db = s.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=0)
    q = torch.from_numpy(oracle.pack(Q).view(np.int64)).cuda()
    m = torch.from_numpy(modes).cuda()
    T = int(np.percentile(exp, 20))
    for threshold in (B.NO_THRESHOLD, T):
        es, ei = oracle.topk(exp, k, threshold)
        sc, ix = s.topk(db, q, m, k, threshold)
        assert np.array_equal(sc.cpu().numpy().view(np.uint32), es) and np.array_equal(ix.cpu().numpy(), ei)
        sc.fill_(7)
        B.fastid_topk_noalloc(s.ctx, db, q, m, k, threshold, sc, ix)
        assert np.array_equal(sc.cpu().numpy().view(np.uint32), es) and np.array_equal(ix.cpu().numpy(), ei)
    for dtype in (torch.int16, torch.int32):
        assert np.array_equal(s.scores(db, q, m, dtype).cpu().numpy().astype(np.int64), exp.astype(np.int64))
    T = int(np.percentile(exp, 2))
    oq, orr, osc = oracle.hits(exp, T)
    hq, hr, hs, hc = s.hits(db, q, m, T, oq.size + 3)
    assert B.fastid_sync_status(s.ctx) == B.OK and int(hc.item()) == oq.size
    n = oq.size
    assert np.array_equal(hq[:n].cpu().numpy(), oq) and np.array_equal(hr[:n].cpu().numpy(), orr)
    assert np.array_equal(hs[:n].cpu().numpy().view(np.uint32), osc)
    db.close()
    s.ctx.close()
