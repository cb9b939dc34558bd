"""Starting cuts of the few-query form: databases around the sample's steps
(a sixteenth of the references, one round of 248, four rounds), samples that
just hold or just miss k references, and calls back to back on one stream (each
kernel of a call begins beside the end of the one before).  Exact integers
against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402


@pytest.fixture(scope="module")
def searcher():
    import __graft_entry__
    __graft_entry__.build()
    s = Searcher(0, B.FORM_TENSOR_FP4_PACKED)
    yield s
    s.ctx.close()


def problem(n_q, n_refs, n_loci, seed):
    rng = np.random.default_rng(seed)
    R = (rng.random((n_refs, n_loci)) < 0.4).astype(np.uint8)
    R[:: max(1, n_refs // 9)] = 0  # (sampled references among the best)
    Q = (rng.random((n_q, n_loci)) < 0.4).astype(np.uint8)
    return R, Q, (rng.random(n_q) < 0.5).astype(np.uint8)


def device(Q, modes):
    return torch.from_numpy(oracle.pack(Q).view(np.int64)).cuda(), torch.from_numpy(modes).cuda()


@pytest.mark.parametrize("n_q", [1, 8, 9])
@pytest.mark.parametrize("n_refs", [15, 16, 127, 128, 511, 512, 513, 3967, 3968, 3969, 15871, 15872, 15873, 31000])
def test_seed_sizes(searcher, n_q, n_refs):
    R, Q, modes = problem(n_q, n_refs, 200, n_refs + n_q)
    db = searcher.load_refs_alleles(torch.from_numpy(R).cuda(), 200, flags=0)
    q, m = device(Q, modes)
    for k in (1, 7, 8, 31, 32):
        sc, ix = searcher.topk(db, q, m, k)
        es, ei = oracle.topk(oracle.select(*oracle.scores(R, Q), modes), k, B.NO_THRESHOLD)
        assert np.array_equal(sc.cpu().numpy().view(np.uint32), es)
        assert np.array_equal(ix.cpu().numpy(), ei)
    db.close()


def test_calls_back_to_back(searcher):
    """Different queries, sizes and databases one after another without a
    wait; every result is its own call's."""
    calls = []
    for i, (n_q, n_refs, n_loci, k) in enumerate([(1, 30000, 300, 5), (40, 30000, 700, 32), (1, 50, 64, 3), (9, 8000, 2048, 16)]):
        R, Q, modes = problem(n_q, n_refs, n_loci, i)
        db = searcher.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=0)
        calls.append((db, *device(Q, modes), k, oracle.topk(oracle.select(*oracle.scores(R, Q), modes), k, B.NO_THRESHOLD)))
    torch.cuda.synchronize()
    got = []
    for _ in range(25):
        for db, q, m, k, _ in calls:
            sc, ix = searcher.topk(db, q, m, k)
            got.append((sc.clone(), ix.clone()))
    assert B.fastid_sync_status(searcher.ctx) == B.OK
    for i, (sc, ix) in enumerate(got):
        es, ei = calls[i % len(calls)][4]
        assert np.array_equal(sc.cpu().numpy().view(np.uint32), es)
        assert np.array_equal(ix.cpu().numpy(), ei)
    for c in calls:
        c[0].close()
