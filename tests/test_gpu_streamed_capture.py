"""Streamed calls captured in a graph, below and above the query count from which
blocks go through an FP4 operand, with that operand and without: captured,
replayed twice and equal to the call itself.  (What a call asks of the context's
memory pool must be allowed while its stream is captured.)"""
import pytest

from host import ctx_hooks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402

# (scores are 480 on average and 15.5 apart: T leaves a few hits in ten thousand)
N_LOCI, N_REFS, BLOCK, K, T = 1000, 30_000, 8192, 10, 430


@pytest.mark.parametrize("fp4", [-1, 0], ids=["own rule", "packed rows"])
@pytest.mark.parametrize("n_q", [20, 200])
def test_streamed_capture(tmp_path, n_q, fp4):
    import __graft_entry__
    __graft_entry__.build()
    g = torch.Generator(device="cuda").manual_seed(n_q)
    rand = lambda n: (torch.rand((n, N_LOCI), device="cuda", generator=g) < 0.4).to(torch.uint8)  # noqa: E731
    s = Searcher(0, B.FORM_AUTO)
    ctx_hooks(tmp_path).hook_fp4_block_bytes(s.ctx.handle, fp4)
    refs = torch.empty((N_REFS, 16), dtype=torch.int64, device="cuda")
    B.fastid_pack(s.ctx, rand(N_REFS), N_LOCI, refs)
    q = torch.empty((n_q, 16), dtype=torch.int64, device="cuda")
    B.fastid_pack(s.ctx, rand(n_q), N_LOCI, q)
    m = torch.zeros(n_q, dtype=torch.uint8, device="cuda")
    host = refs.cpu().pin_memory()
    want = s.topk_streamed(host, N_LOCI, q, m, K, block_refs=BLOCK, flags=0)
    wq, wr, ws, wc = s.hits_streamed(host, N_LOCI, q, m, T, 200_000, block_refs=BLOCK, flags=0)
    torch.cuda.synchronize()
    n = int(wc.item())
    assert 0 < n <= 200_000
    sc, ix = torch.zeros_like(want[0]), torch.zeros_like(want[1])
    hq, hr, hs, hc = (torch.zeros_like(t) for t in (wq, wr, ws, wc))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.fastid_topk_streamed(s.ctx, host, N_LOCI, 0, BLOCK, q, m, K, B.NO_THRESHOLD, sc, ix)
        B.fastid_compare_streamed(s.ctx, host, N_LOCI, 0, BLOCK, q, m, T, hq, hr, hs, hc)
    for _ in range(2):
        for t in (sc, ix, hq, hr, hs, hc):
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert B.fastid_sync_status(s.ctx) == B.OK
        assert torch.equal(sc, want[0]) and torch.equal(ix, want[1])
        assert int(hc.item()) == n
        assert torch.equal(hq[:n], wq[:n]) and torch.equal(hr[:n], wr[:n]) and torch.equal(hs[:n], ws[:n])
    del graph
    s.ctx.close()
