"""The cut shared by a launch's slices, and started from running lists: scores
that tie across slices and across parts keep the lower reference whichever
comes first, running lists that are empty, part full or already better than
everything, k at its ends, in both tensor forms.  Exact integers."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

FORMS = {"fp8": (B.FORM_TENSOR, B.REFS_TENSOR), "fp4": (B.FORM_TENSOR_FP4, B.REFS_FP4),
         "fp4packed": (B.FORM_TENSOR_FP4_PACKED, 0)}


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("n_q,k", [(1, 1), (40, 32), (300, 16)])
def test_cut_from_running_lists(form, n_q, k):
    import __graft_entry__
    __graft_entry__.build()
    n_refs, n_loci = 4096, 12  # a dozen distinct scores: nearly every entry ties
    rng = np.random.default_rng(n_q + k)
    R = (rng.random((n_refs, n_loci)) < 0.5).astype(np.uint8)
    Q = (rng.random((n_q, n_loci)) < 0.5).astype(np.uint8)
    modes = (np.arange(n_q) % 2).astype(np.uint8)
    exp = oracle.select(*oracle.scores(R, Q), modes)
    code, flags = FORMS[form]
    s = Searcher(0, code)
    db = s.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=flags)
    q = torch.from_numpy(oracle.pack(Q).view(np.int64)).cuda()
    m = torch.from_numpy(modes).cuda()
    for parts in ([0, 1, 2, 3], [3, 1, 0, 2]):  # of 1024 rows, in either order
        run_s = torch.full((n_q, k), -1, dtype=torch.int32, device="cuda")
        run_i = torch.full((n_q, k), -1, dtype=torch.int64, device="cuda")
        seen = []
        for p in parts:
            n = 256 if not seen else 1024  # the first call leaves some lists part full when k > its hits
            v = B.fastid_refs_view(s.ctx, db, p * 1024, n)
            B.fastid_topk_accumulate(s.ctx, v, p * 1024, q, m, k, 3 if not seen else n_loci, run_s, run_i)
            v.close()
            rows = np.arange(p * 1024, p * 1024 + n)
            seen.append((rows, 3 if n == 256 else n_loci))
            cols = np.concatenate([r[(exp[:, r] <= t).any(0)] for r, t in seen])
            sc = np.full((n_q, cols.size), oracle.UINT32_MAX, np.uint32)
            for r, t in seen:
                for j in np.nonzero(np.isin(cols, r))[0]:
                    ok = exp[:, cols[j]] <= t
                    sc[ok, j] = exp[ok, cols[j]]
            es, ei = oracle.topk(sc, k, n_loci, ref_ids=cols)
            assert B.fastid_sync_status(s.ctx) == B.OK
            assert np.array_equal(run_s.cpu().numpy().view(np.uint32), es)
            assert np.array_equal(run_i.cpu().numpy(), ei)
    sc, ix = s.topk(db, q, m, k)
    es, ei = oracle.topk(exp, k)
    assert np.array_equal(sc.cpu().numpy().view(np.uint32), es) and np.array_equal(ix.cpu().numpy(), ei)
    db.close()
    s.ctx.close()
