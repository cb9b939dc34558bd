"""The few-query form (up to 64 queries over packed rows, references as the
MMA's M operand in TMEM) at its edges: query counts around the 16-column steps
and the accumulator counts, loci around the 256- and 512-locus chunks and where
the queries stop fitting shared memory, one reference, partial tiles, odd and
even tiles a CTA, queries that explain nothing or everything, ties, thresholds,
views and running lists.  Exact integers against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

# queries, references, loci, k
SHAPES = [(1, 1, 1, 1), (1, 127, 64, 32), (15, 128, 255, 7), (16, 129, 256, 16), (17, 1000, 257, 32), (31, 3000, 511, 1),
          (32, 3000, 512, 10), (33, 3000, 513, 10), (48, 152 * 128, 700, 4), (49, 152 * 128 + 1, 700, 4),
          (63, 152 * 128 * 2 - 5, 1500, 16), (64, 152 * 128 * 3 + 77, 1024, 32), (65, 3000, 1024, 32),
          (3, 152 * 128 * 5, 300, 5), (1, 2000, 16384, 8), (16, 2000, 16384, 32), (17, 1000, 16384, 32),
          (64, 2000, 4600, 32), (2, 1000, 30000, 4)]


@pytest.fixture(scope="module")
def searcher():
    import __graft_entry__
    __graft_entry__.build()
    s = Searcher(0, B.FORM_TENSOR_FP4_PACKED)
    yield s
    s.ctx.close()


def check(s, db, R, Q, modes, k, T=B.NO_THRESHOLD):
    q = torch.from_numpy(oracle.pack(Q).view(np.int64)).cuda()
    sc, ix = s.topk(db, q, torch.from_numpy(modes).cuda(), k, T)
    assert B.fastid_sync_status(s.ctx) == B.OK
    es, ei = oracle.topk(oracle.select(*oracle.scores(R, Q), modes), k, T)
    assert np.array_equal(sc.cpu().numpy().view(np.uint32), es)
    assert np.array_equal(ix.cpu().numpy(), ei)


@pytest.mark.parametrize("n_q,n_refs,n_loci,k", SHAPES)
def test_few_shapes(searcher, n_q, n_refs, n_loci, k):
    rng = np.random.default_rng(n_q * 131 + n_refs + n_loci)
    R = (rng.random((n_refs, n_loci)) < 0.4).astype(np.uint8)
    Q = (rng.random((n_q, n_loci)) < 0.4).astype(np.uint8)
    Q[::3] = R[rng.integers(0, n_refs, len(Q[::3]))]
    Q[n_q - 1] = 1  # explains everything
    modes = (rng.random(n_q) < 0.5).astype(np.uint8)
    db = searcher.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=0)
    check(searcher, db, R, Q, modes, k)
    check(searcher, db, R, Q, modes, k, n_loci // 4)
    check(searcher, db, R, Q, modes, k, 0)
    db.close()


@pytest.mark.parametrize("n_q", [1, 40, 64])
def test_few_ties_and_extremes(searcher, n_q):
    """Twelve loci (nearly every entry of a list ties, far past k), and
    references of all zeros and all ones."""
    n_refs, n_loci = 152 * 128 + 300, 12
    rng = np.random.default_rng(n_q)
    R = (rng.random((n_refs, n_loci)) < 0.5).astype(np.uint8)
    R[5000:9000] = 0
    R[9000:13000] = 1
    Q = (rng.random((n_q, n_loci)) < 0.5).astype(np.uint8)
    Q[0] = 0
    Q[-1] = 1
    modes = (np.arange(n_q) % 2).astype(np.uint8)
    db = searcher.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=0)
    for k in (1, 32):
        check(searcher, db, R, Q, modes, k)
        v = B.fastid_refs_view(searcher.ctx, db, 4864, 9000)
        check(searcher, v, R[4864:13864], Q, modes, k)
        v.close()
    db.close()


def test_few_adverse_order(searcher):
    """References that get better to the last one: every tile refills the
    queues, and no sample or other slice helps."""
    n_loci, n_refs = 600, 40_000
    R = np.zeros((n_refs, n_loci), np.uint8)
    live = np.linspace(n_loci, 0, n_refs).astype(np.int64)
    R[np.arange(n_loci)[None, :] < live[:, None]] = 1
    Q = np.zeros((50, n_loci), np.uint8)
    modes = (np.arange(50) % 2).astype(np.uint8)
    db = searcher.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=0)
    check(searcher, db, R, Q, modes, 32)
    check(searcher, db, R, Q, modes, 3)
    db.close()
