"""Waits inside kernels that are given up (tera_ctx_wait_limit of 0: any wait is):
the call latches TERA_ETIMEOUT, nothing it guards is written, and the next call
with the usual limit is right again."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from synth import Generator, Workload, to_numpy

FILL = 0xA5


@pytest.fixture(scope="module")
def tera():
    import paper_2509_24063_gb300 as t
    return t


def test_wait_limit_is_checked():
    from paper_2509_24063_gb300 import _lib
    lib = _lib.load()
    assert lib.tera_ctx_wait_limit(ctypes.c_void_p(), 1000) == _lib.EINVAL


def until_given_up(tera, ctx, call, clean):
    """Runs call() with no waiting allowed until it has given a wait up (its blocks
    run side by side, so the first run nearly always does); clean() prepares each run."""
    ctx.wait_limit(0)
    for _ in range(50):
        clean()
        call()
        code, _ = ctx.status(raise_on_error=False)
        assert code in (tera.OK, tera.ETIMEOUT)
        if code == tera.ETIMEOUT:
            break
    assert code == tera.ETIMEOUT
    torch.cuda.synchronize()
    ctx.wait_limit(1000000)


@pytest.mark.gpu
@pytest.mark.parametrize("path", ["batched", "all_pairs"])
def test_setup_given_up_writes_no_message(tera, path):
    # 110,592 pairs: 108 blocks of the setup, which wait for one another
    wl = Workload("t", 120000, (0.0,) * 3, (640.0,) * 3, (16, 16, 16), 10.0, 2,
                  p_grow=0.1, p_divide=0.02, p_die=0.02, seed=5)
    states = list(Generator(wl, device="cuda").series(2))
    g = oracle.make_grid(wl.lo, wl.hi, wl.grid, wl.w)
    ctx = tera.Context(wl.lo, wl.hi, wl.grid, wl.w)
    ex = tera.AuraExchange(ctx, max_agents=140000, max_records=300000, path=path)
    ex.step(states[0])
    ctx.status()
    res0 = oracle.exchange_iteration(g, to_numpy(states[0]))
    res = oracle.exchange_iteration(g, to_numpy(states[1]), ref=(res0["ref_next"], res0["pair_off"]),
                                    recv_ref=(res0["recv"], res0["recv_off"]))
    args, kw = ex.codec_args(1)
    ex.part.pair_off = ex.pair_off[1]
    ctx.partition(states[1], ex.part)
    if path == "batched":
        ctx.pack_ids(states[1], ex.part, ex.rec, ex.rec_ids)

        def call():
            ctx.codec_batched(*args, **kw)
    else:
        ctx.pack(states[1], ex.part, ex.rec)

        def call():
            ctx.delta_encode(*args[:8])
    ctx.status()
    outputs = [ex.ref[1], ex.wire, ex.wire_len, ex.recv[1]]

    def fill():
        for t in outputs:
            t.view(torch.uint8).fill_(FILL)

    until_given_up(tera, ctx, call, fill)
    for t in outputs:
        assert bool((t.view(torch.uint8) == FILL).all())
    call()
    if path != "batched":
        ctx.delta_decode(ex.wire, ex.wire_off, *args[8:])
    assert ctx.status(raise_on_error=False)[0] == tera.OK
    np.testing.assert_array_equal(ex.wire_len.cpu().numpy().view(np.uint64), res["wire_len"])
    units = int(res["pair_off"][-1]) + ctx.n_pairs
    for got, want in ((ex.ref[1], res["ref_next"]), (ex.recv[1], res["recv"])):
        assert got[:units * 64].cpu().numpy().tobytes() == want[:units * 64].tobytes()
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("grad", [False, True])
def test_training_given_up_changes_nothing(tera, grad):
    # 1 M samples: 256 chunks of the scan that finds the valid ones' places
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    samples = torch.randn(1 << 20, 12, generator=g, device="cuda")
    samples[:, 11] = (samples[:, 11] > 0).float()
    samples = samples.reshape(-1)
    params = 0.05 * torch.randn(4931, generator=g, device="cuda")
    ctx = tera.Context((0.0,) * 3, (100.0, 100.0, 50.0), (2, 2, 1), 30.0)
    out = torch.empty_like(params)

    def call():
        try:
            ctx.mlp_grad(samples, params, out) if grad else ctx.mlp_train(samples, out, 2, 512, 0.1)
        except tera.TeraError as e:
            assert e.status == tera.ETIMEOUT
            assert bool((out == params).all())

    until_given_up(tera, ctx, call, lambda: out.copy_(params))
    fresh = tera.Context((0.0,) * 3, (100.0, 100.0, 50.0), (2, 2, 1), 30.0)
    results = []
    for c in (ctx, fresh):
        out.copy_(params)
        n = c.mlp_grad(samples, params, out) if grad else c.mlp_train(samples, out, 2, 512, 0.1)
        assert c.status(raise_on_error=False)[0] == tera.OK
        results.append((n, out.clone()))
    assert results[0][0] == results[1][0] and torch.equal(results[0][1], results[1][1])
    ctx.close()
    fresh.close()


@pytest.mark.gpu
def test_partition_given_up_leaves_every_pair_empty(tera):
    # 2 M agents: eight chunks of the scan over the runs, and a sort of many tiles
    n = 1 << 21
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    st = {f: torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 400.0
          for f in ("x", "y", "z", "diameter", "volume", "adherence", "density")}
    st["id"] = torch.arange(n, device="cuda")
    space = ((0.0,) * 3, (400.0,) * 3, (4, 4, 4), 10.0)
    ctx = tera.Context(*space)
    cap = n
    part = tera.PartitionBuffers.allocate(n, ctx.n_pairs, cap, "cuda")
    rec = torch.empty((cap + ctx.n_pairs) * 64, dtype=torch.uint8, device="cuda")

    def call():
        ctx.partition(st, part)
        ctx.pack(st, part, rec)

    until_given_up(tera, ctx, call, lambda: rec.fill_(FILL))
    assert not bool(part.pair_off.any()) and not bool(part.pair_count.any())
    assert bool((rec[ctx.n_pairs * 64:] == FILL).all())  # headers alone
    fresh = tera.Context(*space)
    results = []
    for c in (ctx, fresh):
        rec.fill_(FILL)
        c.partition(st, part)
        c.pack(st, part, rec)
        assert c.status(raise_on_error=False)[0] == tera.OK
        results.append((part.pair_off.clone(), rec.clone()))
    for a, b in zip(*results):
        assert torch.equal(a, b)
    ctx.close()
    fresh.close()
