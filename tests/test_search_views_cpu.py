"""Searcher.build_queries returns a tensor of its own over the searcher's buffer:
what a caller does to that tensor's shape in place does not reach the next
call.  The library's entry points are stubbed; nothing runs on a GPU."""
import pytest

torch = pytest.importorskip("torch")

from paper_1707_00516_gb300 import binding as B  # noqa: E402
from paper_1707_00516_gb300.search import Searcher  # noqa: E402


@pytest.mark.parametrize("change", [lambda q: q.squeeze_(0), lambda q: q.t_(), lambda q: q.unsqueeze_(0),
                                    lambda q: q.resize_(2, 1)])
def test_a_callers_shape_change_stays_the_callers(monkeypatch, change):
    shapes = []
    monkeypatch.setattr(B, "fastid_pack", lambda ctx, a, n_loci, packed: None)
    monkeypatch.setattr(B, "fastid_mix", lambda ctx, src, w, off, out: shapes.append(tuple(out.shape)))
    s = Searcher.__new__(Searcher)
    s.device, s.ctx = torch.device("cpu"), None
    s._pinned, s._devbuf, s._devview = {}, {}, {}
    src, off = torch.zeros((3, 130), dtype=torch.uint8), torch.tensor([0, 3], dtype=torch.int32)
    first = s.build_queries(src, off, 130)
    at = first.data_ptr()
    change(first)
    second = s.build_queries(src, off, 130)
    assert shapes == [(1, 3), (1, 3)]
    assert tuple(second.shape) == (1, 3) and second.is_contiguous() and second.data_ptr() == at
