"""The batched codec's predictions (the network over tiles of 64 slots per warp)
give the bytes of the per-call codec (the network slot by slot), from a few
slots, one part of a tile, to several tiles per warp."""
import numpy as np
import pytest
import torch

from test_gpu_predictor import drift
from synth import Generator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 90, 5000, 33_000, 130_001])
def test_network_tiles(n):
    import paper_2509_24063_gb300 as tera
    wl = drift(n=n, iters=4, seed=n)
    states = list(Generator(wl, device="cuda").series(wl.iterations))
    rng = np.random.default_rng(n)
    params = torch.from_numpy((rng.standard_normal(4931) * 0.1).astype(np.float32)).cuda()
    nmax = max(int(s["x"].shape[0]) for s in states)
    outs = []
    for path in ("all_pairs", "batched"):
        ctx = tera.Context(wl.lo, wl.hi, wl.grid, wl.w)
        ex = tera.AuraExchange(ctx, nmax, 8 * nmax + 1024, path=path, params=params)
        got = []
        for st in states:
            ex.wire.zero_()  # what lies between two messages is not written
            ex.step(st)
            ctx.status()
            got.append((ex.wire_off.clone(), ex.wire[:int(ex.wire_off[-1])].clone()))
        outs.append(got)
        ctx.close()
    for a, b in zip(*outs):
        assert torch.equal(a[0], b[0])
        assert torch.equal(a[1], b[1])
