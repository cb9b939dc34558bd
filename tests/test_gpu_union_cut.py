"""The cut that a launch's slices publish to one another: numbers of slices
below, at and above a group (query counts from one tile to many, unpaired and
paired, with and without a tail), streams long enough that slices publish and
read each other's bounds, k at and around the published rank's steps, running
lists, and best references that all sit in one slice or at its ends.  Exact
integers against the oracle, where nearly every entry ties too."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

FORMS = {"fp8": (B.FORM_TENSOR, B.REFS_TENSOR), "fp4": (B.FORM_TENSOR_FP4, B.REFS_FP4),
         "fp4packed": (B.FORM_TENSOR_FP4_PACKED, 0)}


SHAPES = [(100, 120_000, 64), (130, 60_000, 300), (400, 70_001, 14), (1300, 50_000, 200), (2100, 40_000, 100)]


@pytest.fixture(scope="module", params=SHAPES, ids=lambda p: "x".join(map(str, p)))
def problem(request):
    n_q, n_refs, n_loci = request.param
    rng = np.random.default_rng(n_q)
    R = (rng.random((n_refs, n_loci)) < 0.5).astype(np.uint8)
    R[7000:7100] = R[7000:7100] & (rng.random((100, n_loci)) < 0.1)  # few alleles: the best, side by side
    R[n_refs - 3:] = 0
    Q = (rng.random((n_q, n_loci)) < 0.5).astype(np.uint8)
    Q[::7] = R[rng.integers(0, n_refs, len(Q[::7]))]
    modes = (rng.random(n_q) < 0.5).astype(np.uint8)
    exp = oracle.select(*oracle.scores(R, Q), modes)
    low = np.where(exp <= n_loci // 3, exp, oracle.UINT32_MAX).astype(np.uint32)
    return R, Q, modes, oracle.topk(exp, 32), oracle.topk(low, 32, n_loci // 3)


@pytest.mark.parametrize("form", sorted(FORMS))
def test_union_cut(problem, form):
    import __graft_entry__
    __graft_entry__.build()
    R, Q, modes, (es, ei), (ls, li) = problem
    n_q, (n_refs, n_loci) = len(Q), R.shape
    code, flags = FORMS[form]
    s = Searcher(0, code)
    db = s.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=flags)
    q = torch.from_numpy(oracle.pack(Q).view(np.int64)).cuda()
    m = torch.from_numpy(modes).cuda()
    for k in (2, 3, 11, 16, 17, 32):  # (a shorter list is the longer one's beginning)
        sc, ix = s.topk(db, q, m, k)
        assert np.array_equal(sc.cpu().numpy().view(np.uint32), es[:, :k]), k
        assert np.array_equal(ix.cpu().numpy(), ei[:, :k]), k
    # the database once more, into lists that hold its best already, with a threshold
    run_s, run_i = sc.clone(), ix.clone()
    B.fastid_topk_accumulate(s.ctx, db, n_refs, q, m, 32, n_loci // 3, run_s, run_i)
    assert B.fastid_sync_status(s.ctx) == B.OK
    run_s, run_i = run_s.cpu().numpy().view(np.uint32), run_i.cpu().numpy()
    li = np.where(li >= 0, li + n_refs, np.iinfo(np.int64).max)  # (an unused entry sorts last)
    ei = np.where(ei >= 0, ei, np.iinfo(np.int64).max)
    for r in range(n_q):
        both = sorted(zip(np.concatenate([es[r], ls[r]]).tolist(), np.concatenate([ei[r], li[r]]).tolist()))[:32]
        assert [b[0] for b in both] == run_s[r].tolist()
        assert [b[1] for b in both] == run_i[r].tolist()
    db.close()
