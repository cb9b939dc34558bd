"""Packing of rows at every alignment: row strides and first bytes off 16,
row ends inside a 16-byte block, one row, values other than 0 and 1, and an
allele buffer that ends exactly at its last row.  Exact bits."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1707_00516_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("n", [1, 3, 130])
@pytest.mark.parametrize("n_loci", [1, 15, 16, 17, 63, 65, 127, 1501, 2049])
@pytest.mark.parametrize("first,gap", [(0, 0), (1, 0), (15, 0), (7, 3), (0, 16), (9, 7)])
def test_pack_alignments(n, n_loci, first, gap):
    import __graft_entry__
    __graft_entry__.build()
    rng = np.random.default_rng(n * 10_000 + n_loci * 10 + first)
    ld = n_loci + gap
    flat = rng.integers(0, 256, first + (n - 1) * ld + n_loci).astype(np.uint8)
    flat[rng.random(flat.size) < 0.5] = 0
    dev = torch.from_numpy(flat).cuda()
    rows = torch.as_strided(dev, (n, n_loci), (ld, 1), first)
    A = np.lib.stride_tricks.as_strided(flat[first:], (n, n_loci), (ld, 1))
    words = (n_loci + 63) // 64 + 1
    out = torch.full((n, words), -1, dtype=torch.int64, device="cuda")
    norms = torch.empty(n, dtype=torch.int32, device="cuda")
    ctx = B.Context()
    B.fastid_pack(ctx, rows, n_loci, out, norms)
    exp = oracle.pack((A != 0).astype(np.uint8), ld_words=words)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), exp)
    assert np.array_equal(norms.cpu().numpy(), (A != 0).sum(1))
    ctx.close()
