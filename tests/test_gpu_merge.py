"""The merge of per-slice top-k lists at its edges: list counts around the
warps-per-query steps (8, 9, 33, 152 slices), blocks with idle warps, and
enough queries that fewer warps a query are used.  Few loci, so that most
scores tie and the order rests on the reference index.  Exact integers."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

SHAPES = [(1, 224 * 8, 16), (1, 224 * 9, 32), (17, 224 * 33 - 5, 1), (3, 224 * 152, 32), (2100, 3000, 7), (9000, 500, 3)]


@pytest.mark.parametrize("form", ["plain", "fp4"])
@pytest.mark.parametrize("n_q,n_refs,k", SHAPES)
def test_merge_of_many_lists(form, n_q, n_refs, k):
    import __graft_entry__
    __graft_entry__.build()
    n_loci = 24
    rng = np.random.default_rng(n_q * 7 + n_refs)
    R = (rng.random((n_refs, n_loci)) < 0.4).astype(np.uint8)
    Q = (rng.random((n_q, n_loci)) < 0.4).astype(np.uint8)
    modes = (np.arange(n_q) % 2).astype(np.uint8)
    s = Searcher(0, {"plain": B.FORM_PLAIN, "fp4": B.FORM_TENSOR_FP4}[form])
    db = s.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=B.REFS_FP4 if form == "fp4" else 0)
    q = s.build_queries(torch.from_numpy(Q).cuda(), torch.arange(n_q + 1, dtype=torch.int32, device="cuda"), n_loci)
    sc, ix = s.topk(db, q, torch.from_numpy(modes).cuda(), k)
    rows = np.arange(n_q) if n_q <= 64 else rng.choice(n_q, 64, replace=False)
    mis, une = oracle.scores(R, Q[rows])
    es, ei = oracle.topk(oracle.select(mis, une, modes[rows]), k)
    assert B.fastid_sync_status(s.ctx) == B.OK
    assert np.array_equal(sc.cpu().numpy().view(np.uint32)[rows], es)
    assert np.array_equal(ix.cpu().numpy()[rows], ei)
    db.close()
    s.ctx.close()
