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


@pytest.mark.parametrize("path", ["batched", "all_pairs"])
@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("slots,share", [(16300, 0.3), (16500, 0.3), (16500, 0.0), (60000, 0.02),
                                         (60000, 0.2)])
def test_many_slots_and_a_short_message(slots, share, shuffle, path):
    # nearly every agent gone, or all: slots of a pair round the line above which
    # they are looked up by many blocks
    import paper_2509_24063_gb300 as tera
    from test_gpu_tiles import two_pairs
    first, second, _ = two_pairs(slots, 700, slots)
    g = torch.Generator(device="cuda")
    g.manual_seed(slots)
    k = second["x"].shape[0]
    keep = torch.rand(k, generator=g, device="cuda") < share
    states = [first, {f: v[keep].contiguous() for f, v in second.items()}]
    if shuffle:
        for i, st in enumerate(states):
            perm = torch.randperm(st["x"].shape[0], generator=g, device="cuda")
            states[i] = {f: v[perm].contiguous() for f, v in st.items()}
    run_states(tera, states, (0.0,) * 3, (200.0, 100.0, 100.0), (2, 1, 1), 20.0, path=path)
