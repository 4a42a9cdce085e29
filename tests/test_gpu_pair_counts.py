"""The partition over grids at both sides of the line between its two searches for
the pairs' offsets (16,384 pairs), and where the sort takes two passes of the
full 256 digits, against the oracle's lists."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 70, 30000])
@pytest.mark.parametrize("grid", [(101, 3, 2), (76, 4, 2), (11, 11, 11), (13, 13, 14)])
def test_pair_lists(grid, n):
    import paper_2509_24063_gb300 as tera
    hi = tuple(20.0 * k for k in grid)
    g = torch.Generator(device="cuda")
    g.manual_seed(n + grid[0])
    st = {f: torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * hi[a]
          for a, f in enumerate(("x", "y", "z"))}
    for f in ("diameter", "volume", "adherence", "density"):
        st[f] = torch.ones(n, device="cuda", dtype=torch.float64)
    st["id"] = torch.arange(n, device="cuda")
    ctx = tera.Context((0.0,) * 3, hi, grid, 4.0)
    part = tera.PartitionBuffers.allocate(n, ctx.n_pairs, 3 * n + 64, "cuda")
    ctx.partition(st, part)
    assert ctx.status(raise_on_error=False)[0] == tera.OK
    og = oracle.make_grid((0.0,) * 3, hi, grid, 4.0)
    code, owner, mask = oracle.classify(og, *(st[f].cpu().numpy() for f in "xyz"))
    assert code == oracle.OK
    _, cnt, off, idx = oracle.pair_lists(og, owner, mask)
    total = int(off[-1])
    np.testing.assert_array_equal(part.pair_off.cpu().numpy().view(np.uint64), off)
    np.testing.assert_array_equal(part.pair_count.cpu().numpy().view(np.uint64), cnt)
    np.testing.assert_array_equal(part.pair_idx.cpu().numpy().view(np.uint32)[:total], idx[:total])
    ctx.close()
