"""The first calls of a context on a stream of the caller's own (non-blocking: it
does not wait for the default stream, on which new scratch is cleared), with
more than 1,024 pairs, whose setup blocks read cleared words; byte for byte
against the oracle.  The allocations are made where a freed buffer of set bits
lay."""
import pytest
import torch

import oracle
from synth import Generator, Workload, to_numpy
from test_gpu_parity import compare_iteration

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["batched", "all_pairs"])
@pytest.mark.parametrize("tune", [None, (256, 4, 0, 0)])
def test_first_call_on_another_stream(path, tune):
    import paper_2509_24063_gb300 as tera
    wl = Workload("t", 60000, (0.0,) * 3, (500.0,) * 3, (10, 10, 10), 12.0, 2,
                  p_grow=0.1, p_divide=0.02, p_die=0.02, seed=41)
    states = list(Generator(wl, device="cuda").series(2))
    g = oracle.make_grid(wl.lo, wl.hi, wl.grid, wl.w)
    for _ in range(3):
        ctx = tera.Context(wl.lo, wl.hi, wl.grid, wl.w)
        ex = tera.AuraExchange(ctx, max_agents=80000, max_records=200000, path=path, tune=tune)
        dirty = torch.empty(1 << 28, dtype=torch.uint8, device="cuda").fill_(0xFF)
        torch.cuda.synchronize()
        del dirty
        torch.cuda.empty_cache()
        own = torch.cuda.Stream()
        ref = recv_ref = None
        for st in states:
            ex.step(st, own)
            assert ctx.status(own, raise_on_error=False)[0] == tera.OK
            res = oracle.exchange_iteration(g, to_numpy(st), ref=ref, recv_ref=recv_ref)
            compare_iteration(ctx, ex, st, res, ctx.n_pairs)
            ref, recv_ref = (res["ref_next"], res["pair_off"]), (res["recv"], res["recv_off"])
        ctx.close()
