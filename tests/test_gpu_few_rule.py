"""Top-k over packed rows on both sides of the few-query form's rule (33 to 64
queries take it over a long database only): a database of 700 MB and views just
below and above its two lines, against the plain form and the FP4 copy, which
the rule does not concern.  Identical lists."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

N = 2048
ROWS = {"short": 1000, "48-": (320 << 20) // 256 - 1, "48": (320 << 20) // 256, "64-": (640 << 20) // 256 - 1, "all": 2_700_000}


@pytest.fixture(scope="module")
def db():
    import __graft_entry__
    __graft_entry__.build()
    s = Searcher(0, B.FORM_TENSOR_FP4_PACKED)
    g = torch.Generator(device="cuda").manual_seed(3)
    rows = torch.randint(-2**63, 2**63 - 1, (ROWS["all"], N // 64), dtype=torch.int64, device="cuda", generator=g)
    db = s.load_refs_packed(rows, N, flags=B.REFS_FP4)
    yield s, db, rows
    db.close()
    s.ctx.close()


@pytest.mark.parametrize("rows", sorted(ROWS))
@pytest.mark.parametrize("n_q", [32, 33, 40, 48, 49, 64, 65])
def test_few_rule(db, rows, n_q):
    s, base, packed = db
    g = torch.Generator(device="cuda").manual_seed(n_q)
    q = torch.randint(-2**63, 2**63 - 1, (n_q, N // 64), dtype=torch.int64, device="cuda", generator=g)
    q[::4] = packed[torch.randint(0, ROWS[rows], (len(q[::4]),), device="cuda", generator=g)]
    m = (torch.arange(n_q, device="cuda") % 2).to(torch.uint8)
    view = B.fastid_refs_view(s.ctx, base, 0, ROWS[rows]) if rows != "all" else base
    for k in (10, 32):
        got = {}
        for form in (B.FORM_TENSOR_FP4_PACKED, B.FORM_TENSOR_FP4, B.FORM_PLAIN):
            B.fastid_set_form(s.ctx, form)
            sc, ix = s.topk(view, q, m, k)
            got[form] = (sc.clone(), ix.clone())
        assert B.fastid_sync_status(s.ctx) == B.OK
        first = got[B.FORM_TENSOR_FP4_PACKED]
        for form in got:
            assert torch.equal(first[0], got[form][0]) and torch.equal(first[1], got[form][1])
    if view is not base:
        view.close()
