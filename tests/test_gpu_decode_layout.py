"""The per-call decode's receive layout and records agree with the batched
codec's, from one box to more pairs than one pass of the layout's block."""
import pytest
import torch

from synth import Generator, Workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["all_pairs", "per_subdomain"])
@pytest.mark.parametrize("grid", [(1, 1, 1), (19, 2, 1), (7, 7, 7)])
def test_layout(grid, path):
    import paper_2509_24063_gb300 as tera
    hi = tuple(20.0 * g for g in grid)
    wl = Workload("t", 6000, (0.0,) * 3, hi, grid, 4.0, 3, p_grow=0.1, p_divide=0.02, p_die=0.02,
                  seed=5)
    states = list(Generator(wl, device="cuda").series(wl.iterations))
    nmax = max(int(s["x"].shape[0]) for s in states)
    outs = []
    for p in (path, "batched"):
        ctx = tera.Context(wl.lo, wl.hi, wl.grid, wl.w, periodic=wl.periodic)
        ex = tera.AuraExchange(ctx, nmax, 27 * nmax, path=p)
        got = []
        for t, st in enumerate(states):
            ex.step(st)
            ctx.status()
            slot = ex.slot_of(t)
            off = ex.recv_off[slot].clone()
            n = (int(off[-1]) + ctx.n_pairs) * 64
            got.append((off, ex.recv[slot][:n].clone()))
        outs.append(got)
        ctx.close()
    for a, b in zip(*outs):
        assert torch.equal(a[0], b[0])
        # the order of a message's records is the reference's on both
        assert torch.equal(a[1], b[1])
