"""Messages with many records that no reference slot has, in pairs matched by a
warp, by a block and through global memory: the tiles the match adds.  Byte for
byte against the oracle; with the predictor's histories the same messages."""
import pytest
import torch

from synth import Generator, Workload
from test_gpu_tiles import run_states

pytestmark = pytest.mark.gpu


def states_of(n, grid, share, seed, side=50.0, w=6.0):
    hi = tuple(side * k for k in grid)
    wl = Workload("t", n, (0.0,) * 3, hi, grid, w, 2, p_grow=0.1, seed=seed)
    first, second = Generator(wl, device="cuda").series(2)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    k = second["x"].shape[0]
    other = torch.rand(k, generator=g, device="cuda") < share
    second["id"] = torch.where(other, second["id"] + 10 * k, second["id"])
    return wl, [first, second]


@pytest.mark.parametrize("path", ["batched", "all_pairs"])
@pytest.mark.parametrize("share", [0.1, 0.5, 1.0])
@pytest.mark.parametrize("n,grid", [(3000, (2, 2, 1)), (60000, (8, 8, 8)), (90000, (2, 1, 1)),
                                    (400000, (2, 1, 1))])
def test_new_records(n, grid, share, path):
    import paper_2509_24063_gb300 as tera
    wl, states = states_of(n, grid, share, 31, w=24.0 if grid == (2, 1, 1) else 6.0)
    run_states(tera, states, wl.lo, wl.hi, wl.grid, wl.w, path=path)


@pytest.mark.parametrize("n,grid", [(60000, (8, 8, 8)), (90000, (2, 1, 1))])
def test_new_records_with_histories(n, grid):
    import paper_2509_24063_gb300 as tera
    wl, states = states_of(n, grid, 0.7, 32, w=24.0 if grid == (2, 1, 1) else 6.0)
    out = []
    for predictor in (False, True):
        ctx = tera.Context(wl.lo, wl.hi, wl.grid, wl.w)
        ex = tera.AuraExchange(ctx, max_agents=n, max_records=3 * n, path="batched",
                               predictor=predictor)
        for st in states:
            ex.step(st)
            assert ctx.status(raise_on_error=False)[0] == tera.OK
        units = int(ex.pair_off[ex.last][-1]) + ctx.n_pairs
        out.append([t.clone() for t in (ex.wire_len, ex.sender_ref()[0][:units * 64],
                                        ex.receiver_ref()[0][:units * 64])])
        ctx.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
