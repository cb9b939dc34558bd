"""Full-matrix stores at their edges: rows that start on 16 bytes and rows
that do not (odd strides, a shifted base), columns ending inside a 32-column
block, one query, query counts around the 32 rows of a warp and the tiles of a
pair, both output widths, in every tensor operand.  Exact integers."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher, words64  # noqa: E402

FORMS = {"fp8": (B.FORM_TENSOR, B.REFS_TENSOR), "fp8packed": (B.FORM_TENSOR_PACKED, 0),
         "fp4": (B.FORM_TENSOR_FP4, B.REFS_FP4), "fp4packed": (B.FORM_TENSOR_FP4_PACKED, 0)}
# queries, references, row stride beyond the references, elements before the first row
CASES = [(1, 1, 0, 0), (1, 224, 0, 0), (31, 225, 0, 0), (33, 449, 7, 0), (64, 512, 8, 0), (129, 1000, 0, 1),
         (300, 703, 1, 0), (300, 704, 0, 8)]


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("n_q,n_refs,extra,shift", CASES)
def test_scores_store(form, n_q, n_refs, extra, shift):
    import __graft_entry__
    __graft_entry__.build()
    n_loci = 300
    rng = np.random.default_rng(n_q * 1000 + n_refs)
    R = (rng.random((n_refs, n_loci)) < 0.5).astype(np.uint8)
    Q = (rng.random((n_q, n_loci)) < 0.5).astype(np.uint8)
    modes = (rng.random(n_q) < 0.5).astype(np.uint8)
    mis, une = oracle.scores(R, Q)
    exp = oracle.select(mis, une, modes)
    code, flags = FORMS[form]
    s = Searcher(0, code)
    db = s.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=flags)
    q = torch.empty((n_q, words64(n_loci)), dtype=torch.int64, device="cuda")
    B.fastid_pack(s.ctx, torch.from_numpy(Q).cuda(), n_loci, q)
    ld = n_refs + extra
    for dtype in (torch.int16, torch.int32):
        flat = torch.full((shift + n_q * ld + 16,), -7, dtype=dtype, device="cuda")
        out = flat[shift:shift + n_q * ld].view(n_q, ld)
        B.fastid_scores(s.ctx, db, q, torch.from_numpy(modes).cuda(), out[:, :n_refs] if n_q > 1 else out)
        got = out.cpu().numpy()
        assert B.fastid_sync_status(s.ctx) == B.OK
        assert np.array_equal(got[:, :n_refs].astype(np.int64), exp.astype(np.int64))
        assert (got[:, n_refs:] == -7).all()  # nothing outside the matrix is written
        assert (flat[:shift] == -7).all() and (flat[shift + n_q * ld:] == -7).all()
    db.close()
    s.ctx.close()
