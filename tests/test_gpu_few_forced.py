"""The few-query form at its edges with the form forced: the rule that chooses
it leaves short databases to the tensor kernel from 33 queries on, so its wider
shapes (48 and 64 columns; 64 is the one with two accumulators) would otherwise
be met by long databases only.  Odd numbers of 256-locus chunks, the fewest
packed stages, one and partial tiles, odd and even tiles a CTA, mass ties, a
stream that keeps the candidate rings full, views, running lists and calls back
to back, each with the form's own shape asserted.  Exact integers against the
oracle."""
import numpy as np
import pytest

import oracle
from host import ctx_hooks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

TILES = 152 * 128  # a reference tile a CTA


@pytest.fixture(scope="module")
def few(tmp_path_factory):
    import __graft_entry__
    __graft_entry__.build()
    hooks = ctx_hooks(tmp_path_factory.mktemp("hooks"))
    s = Searcher(0, B.FORM_TENSOR_FP4_PACKED)
    hooks.hook_few_rule(s.ctx.handle, 1)
    yield s, hooks
    s.ctx.close()


def rows(rng, n, n_loci, p=0.4):
    return (rng.random((n, n_loci)) < p).astype(np.uint8)


def device(Q, modes):
    return torch.from_numpy(oracle.pack(Q).view(np.int64)).cuda(), torch.from_numpy(modes).cuda()


def load(s, R):
    return s.load_refs_alleles(torch.from_numpy(R).cuda(), R.shape[1], flags=0)


def same(sc, ix, es, ei):
    assert np.array_equal(sc.cpu().numpy().view(np.uint32), es)
    assert np.array_equal(ix.cpu().numpy(), ei)


def check(few, db, R, Q, modes, k, T=B.NO_THRESHOLD):
    s, hooks = few
    assert hooks.hook_few_stages(len(Q), R.shape[1], k) > 0
    q, m = device(Q, modes)
    sc, ix = s.topk(db, q, m, k, T)
    assert B.fastid_sync_status(s.ctx) == B.OK
    same(sc, ix, *oracle.topk(oracle.select(*oracle.scores(R, Q), modes), k, T))


@pytest.mark.parametrize("n_q", [16, 33, 47, 48, 49, 63, 64])
@pytest.mark.parametrize("n_refs,n_loci,k", [(1, 1, 1), (127, 64, 32), (129, 257, 16), (3000, 513, 10), (TILES + 1, 700, 4),
                                             (2 * TILES - 5, 1100, 16), (3 * TILES + 77, 256, 32)])
def test_forced_shapes(few, n_q, n_refs, n_loci, k):
    rng = np.random.default_rng(n_q * 131 + n_refs + n_loci)
    R, Q = rows(rng, n_refs, n_loci), rows(rng, n_q, n_loci)
    Q[::3] = R[rng.integers(0, n_refs, len(Q[::3]))]
    Q[n_q - 1] = 1  # explains everything
    modes = (rng.random(n_q) < 0.5).astype(np.uint8)
    db = load(few[0], R)
    check(few, db, R, Q, modes, k)
    check(few, db, R, Q, modes, k, n_loci // 4)
    db.close()


@pytest.mark.parametrize("k", [1, 32])
@pytest.mark.parametrize("n_q", [1, 17, 33, 49])
def test_fewest_stages(few, n_q, k):
    """The most loci that the form takes, which leave it the fewest stages."""
    hooks = few[1]
    fits = [c for c in range(1, 257) if hooks.hook_few_stages(n_q, 256 * c, k) > 0]
    n_loci = 256 * max(fits) - 3
    if max(fits) < 256:
        assert hooks.hook_few_stages(n_q, n_loci, k) == min(hooks.hook_few_stages(n_q, 256 * c, k) for c in fits) <= 6
    rng = np.random.default_rng(n_q + k)
    R, Q = rows(rng, 700, n_loci), rows(rng, n_q, n_loci)
    Q[0] = R[699]
    db = load(few[0], R)
    check(few, db, R, Q, (np.arange(n_q) % 2).astype(np.uint8), k)
    db.close()


@pytest.mark.parametrize("n_q", [8, 32, 48, 64])
def test_forced_ties(few, n_q):
    """Twelve loci: nearly every entry of a list ties, far past k."""
    n_refs, n_loci = TILES + 300, 12
    rng = np.random.default_rng(n_q)
    R, Q = rows(rng, n_refs, n_loci, 0.5), rows(rng, n_q, n_loci, 0.5)
    R[5000:9000] = 0
    R[9000:13000] = 1
    Q[0], Q[-1] = 0, 1
    modes = (np.arange(n_q) % 2).astype(np.uint8)
    db = load(few[0], R)
    for k in (1, 32):
        check(few, db, R, Q, modes, k)
        v = B.fastid_refs_view(few[0].ctx, db, 4864, 9000)
        check(few, v, R[4864:13864], Q, modes, k)
        v.close()
    db.close()


@pytest.mark.parametrize("n_q", [1, 16, 32, 48, 64])
def test_forced_adverse_order(few, n_q):
    """References that get better to the last one: every tile's are candidates
    of every query, the rings stay full and no sample or other slice helps."""
    n_loci, n_refs = 600, 40_000
    R = np.zeros((n_refs, n_loci), np.uint8)
    live = np.linspace(n_loci, 0, n_refs).astype(np.int64)
    R[np.arange(n_loci)[None, :] < live[:, None]] = 1
    Q = np.zeros((n_q, n_loci), np.uint8)
    modes = (np.arange(n_q) % 2).astype(np.uint8)
    db = load(few[0], R)
    for k in (1, 3, 32):
        check(few, db, R, Q, modes, k)
    db.close()


@pytest.mark.parametrize("n_q", [32, 48, 64])
@pytest.mark.parametrize("k", [1, 16, 32])
def test_forced_running_lists(few, n_q, k):
    """Lists kept over three databases, empty at first: equal to one search of
    all of them, and the second and third start from the running k-th."""
    s, hooks = few
    assert hooks.hook_few_stages(n_q, 300, k) > 0
    rng = np.random.default_rng(n_q + k)
    R, Q = rows(rng, 9000, 300), rows(rng, n_q, 300)
    R[4000:4100] = R[100:200]  # ties between databases
    Q[::5] = R[rng.integers(0, 9000, len(Q[::5]))]
    modes = (np.arange(n_q) % 2).astype(np.uint8)
    q, m = device(Q, modes)
    sc = torch.full((n_q, k), -1, dtype=torch.int32, device="cuda")
    ix = torch.full((n_q, k), -1, dtype=torch.int64, device="cuda")
    for lo, hi in ((0, 10), (10, 4000), (4000, 9000)):
        db = load(s, R[lo:hi])
        B.fastid_topk_accumulate(s.ctx, db, lo, q, m, k, B.NO_THRESHOLD, sc, ix)
        assert B.fastid_sync_status(s.ctx) == B.OK
        db.close()
    same(sc, ix, *oracle.topk(oracle.select(*oracle.scores(R, Q), modes), k, B.NO_THRESHOLD))


def test_forced_back_to_back(few):
    """Different queries, sizes and databases one after another without a wait."""
    s, hooks = few
    calls = []
    for i, (n_q, n_refs, n_loci, k) in enumerate([(64, 30000, 300, 5), (40, 30000, 700, 32), (50, 50, 64, 3), (33, 8000, 2048, 16)]):
        assert hooks.hook_few_stages(n_q, n_loci, k) > 0
        rng = np.random.default_rng(i)
        R, Q = rows(rng, n_refs, n_loci), rows(rng, n_q, n_loci)
        modes = (rng.random(n_q) < 0.5).astype(np.uint8)
        calls.append((load(s, R), *device(Q, modes), k, oracle.topk(oracle.select(*oracle.scores(R, Q), modes), k, B.NO_THRESHOLD)))
    torch.cuda.synchronize()
    got = [s.topk(db, q, m, k) for _ in range(25) for db, q, m, k, _ in calls]
    assert B.fastid_sync_status(s.ctx) == B.OK
    for i, (sc, ix) in enumerate(got):
        same(sc, ix, *calls[i % len(calls)][4])
    for c in calls:
        c[0].close()
