"""The partition's scan, sort and pair search at the edges of their tiles, and
with one, two and three digit passes, byte for byte against the oracle."""
import pytest
import torch

import oracle
from synth import Generator, Workload, to_numpy
from test_gpu_parity import compare_iteration

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tera():
    import paper_2509_24063_gb300 as t
    return t


def one_iteration(tera, st, lo, hi, grid, w, max_records):
    ctx = tera.Context(lo, hi, grid, w)
    ex = tera.AuraExchange(ctx, max_agents=int(st["x"].shape[0]), max_records=max_records,
                           path="batched")
    for _ in range(2):  # the second finds the scratch as the first left it
        ex.reset()
        ex.step(st)
        code, _ = ctx.status(raise_on_error=False)
        assert code == tera.OK
        res = oracle.exchange_iteration(oracle.make_grid(lo, hi, grid, w), to_numpy(st))
        compare_iteration(ctx, ex, st, res, ctx.n_pairs)
    ctx.close()
    return int(res["pair_off"][-1])


@pytest.mark.parametrize("entries", [1, 3071, 3072, 3073, 6144, 9217, 400001])
def test_entries_round_a_sort_tile(tera, entries):
    # two boxes, every agent in the other's aura: as many entries as agents
    g = torch.Generator(device="cuda")
    g.manual_seed(entries)

    def rand():
        return torch.rand(entries, generator=g, device="cuda", dtype=torch.float64)

    st = dict(id=torch.arange(entries, device="cuda"), x=85 + 30 * rand(), y=100 * rand(),
              z=100 * rand(), diameter=rand(), volume=rand(), adherence=rand(), density=rand())
    got = one_iteration(tera, st, (0.0,) * 3, (200.0, 100.0, 100.0), (2, 1, 1), 20.0, entries + 7)
    assert got == entries


# runs of 64 agents, 4096 to a chunk of the scan; one, two and three passes of
# the sort (boxes times 27 keys)
@pytest.mark.parametrize("n,grid", [(262143, (4, 4, 4)), (262144, (2, 2, 2)), (262145, (8, 8, 8)),
                                    (30000, (14, 14, 14)), (5000, (3, 1, 2)), (1, (14, 14, 14))])
def test_agents_round_a_scan_chunk_and_key_ranges(tera, n, grid):
    hi = tuple(50.0 * k for k in grid)
    wl = Workload("t", n, (0.0,) * 3, hi, grid, 6.0, 1, seed=n)
    st = next(iter(Generator(wl, device="cuda").series(1)))
    one_iteration(tera, st, wl.lo, wl.hi, wl.grid, wl.w, 3 * n + 1024)
