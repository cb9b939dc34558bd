"""Every kind of call captured into a CUDA graph and replayed, alone and twice in
one graph (a call's first kernel follows another call's last, its later ones
begin beside the end of the one before), on new queries written in place.
Exact integers against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

FORMS = {"plain": (B.FORM_PLAIN, 0), "fp8": (B.FORM_TENSOR, B.REFS_TENSOR), "fp4": (B.FORM_TENSOR_FP4, B.REFS_FP4),
         "fp4packed": (B.FORM_TENSOR_FP4_PACKED, 0)}


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("n_q", [3, 200])
def test_captured_calls(form, n_q):
    import __graft_entry__
    __graft_entry__.build()
    n_refs, n_loci, k, T = 9000, 300, 8, 100
    rng = np.random.default_rng(n_q)
    R = (rng.random((n_refs, n_loci)) < 0.4).astype(np.uint8)
    code, flags = FORMS[form]
    s = Searcher(0, code)
    db = s.load_refs_alleles(torch.from_numpy(R).cuda(), n_loci, flags=flags)
    batches = []
    for _ in range(3):
        Q = (rng.random((n_q, n_loci)) < 0.4).astype(np.uint8)
        modes = (rng.random(n_q) < 0.5).astype(np.uint8)
        batches.append((torch.from_numpy(oracle.pack(Q).view(np.int64)).cuda(), torch.from_numpy(modes).cuda(),
                        oracle.select(*oracle.scores(R, Q), modes)))
    q, m = batches[0][0].clone(), batches[0][1].clone()
    sc, ix = (torch.empty((n_q, k), dtype=t, device="cuda") for t in (torch.int32, torch.int64))
    full = torch.empty((n_q, n_refs), dtype=torch.int16, device="cuda")
    cap = n_q * n_refs
    hq, hr = (torch.empty(cap, dtype=torch.int64, device="cuda") for _ in range(2))
    hs, hn = torch.empty(cap, dtype=torch.int32, device="cuda"), torch.empty(1, dtype=torch.int64, device="cuda")

    def calls():
        B.fastid_topk(s.ctx, db, q, m, k, B.NO_THRESHOLD, sc, ix)
        B.fastid_scores(s.ctx, db, q, m, full)
        B.fastid_compare(s.ctx, db, q, m, T, hq, hr, hs, hn)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        calls()
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
        calls()
    for bq, bm, exp in batches[1:]:
        q.copy_(bq)
        m.copy_(bm)
        for t in (sc, ix, full, hq, hr, hs, hn):
            t.fill_(-1)
        graph.replay()
        torch.cuda.synchronize()
        assert B.fastid_sync_status(s.ctx) == B.OK
        es, ei = oracle.topk(exp, k)
        assert np.array_equal(sc.cpu().numpy().view(np.uint32), es) and np.array_equal(ix.cpu().numpy(), ei)
        assert np.array_equal(full.cpu().numpy().view(np.uint16), exp.astype(np.uint16))
        eq, er = np.nonzero(exp <= T)
        n = int(hn.item())
        assert n == eq.size
        assert np.array_equal(hq[:n].cpu().numpy(), eq) and np.array_equal(hr[:n].cpu().numpy(), er)
        assert np.array_equal(hs[:n].cpu().numpy().view(np.uint32), exp[eq, er])
    del graph
    db.close()
    s.ctx.close()
