"""The hit list's order at the sort's edges: no hits, one, counts around a
tile (4096), more tiles than blocks (256), buffers larger and smaller than the
count, one query holding every hit, and key widths of two and four passes.
Exact integers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

# queries, references, references that every query hits
CASES = [(1, 300, 0), (1, 300, 1), (1, 5000, 4095), (1, 5000, 4096), (1, 5000, 4097), (7, 5000, 586), (64, 40_000, 516),
         (1, 1_300_000, 1_100_000), (300, 70_000, 8333)]


@pytest.mark.parametrize("form", ["plain", "fp4"])
@pytest.mark.parametrize("n_q,n_refs,group", CASES)
def test_hit_order(form, n_q, n_refs, group):
    import __graft_entry__
    __graft_entry__.build()
    n_loci = 64
    rows = np.sort(np.random.default_rng(n_q + group).choice(n_refs, group, replace=False))
    R = np.zeros((n_refs, n_loci), np.uint8)
    R[:, 0] = 1  # one allele that no query explains, except in the group
    R[rows, 0] = 0
    s = Searcher(0, {"plain": B.FORM_PLAIN, "fp4": B.FORM_TENSOR_FP4}[form])
    db = s.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=B.REFS_FP4 if form == "fp4" else 0)
    q = torch.zeros((n_q, 1), dtype=torch.int64, device="cuda")
    modes = torch.ones(n_q, dtype=torch.uint8, device="cuda")
    n = n_q * group
    for cap in sorted({max(1, n), n + 1000, max(1, n // 2)}):
        hq, hr, hs, hc = s.hits(db, q, modes, 0, cap)
        torch.cuda.synchronize()
        assert B.fastid_sync_status(s.ctx) == (B.EOVERFLOW if n > cap else B.OK)
        assert int(hc.item()) == n
        live = min(n, cap)
        hq, hr, hs = hq[:live].cpu().numpy(), hr[:live].cpu().numpy(), hs[:live].cpu().numpy()
        assert not hs.any()
        if n <= cap:
            assert np.array_equal(hq, np.repeat(np.arange(n_q), group)) and np.array_equal(hr, np.tile(rows, n_q))
        else:  # some of the hits, each once, in order
            assert (np.diff(hq * n_refs + hr) > 0).all() and np.isin(hr, rows).all()
    db.close()
    s.ctx.close()
