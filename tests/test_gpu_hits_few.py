"""Hit lists of few hits, which one block sorts: counts around a warp and around
the block's limit (512), buffers that just hold them and smaller ones, queries
and references in many orders, scores that travel with their hits.  Against the
oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402


@pytest.mark.parametrize("form", [B.FORM_PLAIN, B.FORM_AUTO])
@pytest.mark.parametrize("hits", [0, 1, 2, 31, 33, 511, 512, 513])
def test_few_hits(form, hits):
    import __graft_entry__
    __graft_entry__.build()
    n_q, n_refs, n_loci = 40, 6000, 200
    rng = np.random.default_rng(hits)
    R = (rng.random((n_refs, n_loci)) < 0.5).astype(np.uint8)
    Q = (rng.random((n_q, n_loci)) < 0.5).astype(np.uint8)
    pairs = rng.choice(n_refs, hits, replace=False)
    for i, r in enumerate(pairs):  # a copy of a query with a few alleles changed
        R[r] = Q[rng.integers(0, n_q)]
        R[r, rng.choice(n_loci, rng.integers(0, 9), replace=False)] ^= 1
    modes = np.zeros(n_q, np.uint8)
    exp = oracle.select(*oracle.scores(R, Q), modes)
    T = 8
    oq, orr, osc = oracle.hits(exp, T)
    assert oq.size == hits
    s = Searcher(0, form)
    db = s.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci)
    q = torch.from_numpy(oracle.pack(Q).view(np.int64)).cuda()
    m = torch.from_numpy(modes).cuda()
    for cap in sorted({max(1, hits), hits + 3000, max(1, hits // 2)}):
        hq, hr, hs, hc = s.hits(db, q, m, T, cap)
        assert B.fastid_sync_status(s.ctx) == (B.EOVERFLOW if hits > cap else B.OK)
        assert int(hc.item()) == hits
        live = min(hits, cap)
        gq, gr, gs = hq[:live].cpu().numpy(), hr[:live].cpu().numpy(), hs[:live].cpu().numpy().view(np.uint32)
        if hits <= cap:
            assert np.array_equal(gq, oq) and np.array_equal(gr, orr) and np.array_equal(gs, osc)
        else:  # some of the hits, each once, in order
            assert (np.diff(gq * n_refs + gr) > 0).all() and np.array_equal(gs, exp[gq, gr])
    db.close()
    s.ctx.close()
