"""Migration of agents that sit on, beside and far from the edges of their
boxes, byte for byte with the oracle: the kernel decides most agents by the
high words of the coordinates, which say nothing about a coordinate that shares
its word with an edge."""
import numpy as np
import pytest
import torch

import oracle

from test_gpu_migrate import FIELDS, compare, to_dev

pytestmark = pytest.mark.gpu


def edge_values(edges, rng, n):
    """Values on the edges, one and many units in the last place beside them,
    zeros of both signs, subnormals and the midpoints, inside [lo, hi)."""
    lo, hi = edges[0], edges[-1]
    v = [e for e in edges]
    for e in edges:
        v += [np.nextafter(e, -np.inf), np.nextafter(e, np.inf)]
        v += [e + s * 2.0 ** -k for k in (10, 18, 19, 20, 21, 30) for s in (-1.0, 1.0)]
    v += [0.0, -0.0, 5e-324, -5e-324, 1e-300, -1e-300]
    v += list((np.asarray(edges[1:]) + np.asarray(edges[:-1])) / 2)
    v = np.asarray([q for q in v if lo <= q < hi])
    return v[rng.integers(0, len(v), n)]


@pytest.mark.parametrize("periodic", [0, 5])
@pytest.mark.parametrize("n", [1, 255, 257, 2049, 40_001])
def test_box_edges(n, periodic):
    import paper_2509_24063_gb300 as tera
    rng = np.random.default_rng(n + periodic)
    lo, hi, grid, w = (-8.0, -3.0, 1.0), (8.0, 6.0, 2.0), (4, 3, 3), 0.125
    g = oracle.make_grid(lo, hi, grid, w, periodic)
    edges = [[lo[a] + (hi[a] - lo[a]) * i / grid[a] for i in range(grid[a] + 1)] for a in range(3)]
    h = {k: np.ascontiguousarray(rng.random(n)) for k in FIELDS}
    h["id"] = rng.integers(0, 2 ** 62, n).astype(np.uint64)
    for a, k in enumerate("xyz"):
        h[k] = np.ascontiguousarray(edge_values(edges[a], rng, n))
    # boxes before the move: most agents where they are, one in eight elsewhere,
    # and box 5 empty
    status, own, _ = oracle.classify(g, h["x"], h["y"], h["z"])
    assert status == oracle.OK
    nb = int(np.prod(grid))
    prev = np.where(rng.random(n) < 0.125, rng.integers(0, nb, n), own)
    prev = np.where(prev == 5, 6, prev)
    perm = np.argsort(prev, kind="stable")
    h = {k: np.ascontiguousarray(v[perm]) for k, v in h.items()}
    off = np.zeros(nb + 1, dtype=np.uint64)
    off[1:] = np.cumsum(np.bincount(prev, minlength=nb))
    res = oracle.migrate(g, h, off)
    ctx = tera.Context(lo, hi, grid, w, periodic=periodic)
    mig = tera.Migration(ctx, n, max_leavers=n)
    nxt, bo = mig.step(to_dev(h), torch.from_numpy(off.view(np.int64)).cuda())
    code, _ = ctx.status(raise_on_error=False)
    assert code == tera.OK
    compare(mig, res, nxt, bo, n, ctx.n_pairs)
    ctx.close()
