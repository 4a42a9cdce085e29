"""tera_ctx_reserve covers the encode of every pair over tiles: it allocates nothing
more and can be captured at once; a captured encode without that scratch takes
the launches that need none.  Same bytes as the oracle either way."""
import numpy as np
import pytest
import torch

import oracle
from synth import Generator, Workload, to_numpy

pytestmark = pytest.mark.gpu


def encode_case(reserve):
    import paper_2509_24063_gb300 as tera
    wl = Workload("t", 40000, (0.0,) * 3, (160.0,) * 3, (4, 4, 4), 12.0, 1, seed=13)
    st = next(iter(Generator(wl, device="cuda").series(1)))
    ctx = tera.Context(wl.lo, wl.hi, wl.grid, wl.w)
    P, cap = ctx.n_pairs, 120000
    if reserve:
        ctx.reserve(50000, cap)
    part = tera.PartitionBuffers.allocate(50000, P, cap, "cuda")
    u8 = dict(dtype=torch.uint8, device="cuda")
    rec, ref = (torch.empty((cap + P) * 64, **u8) for _ in range(2))
    wire = torch.empty(80 * P + 72 * cap + 64, **u8)
    wire_off = torch.zeros(P + 1, dtype=torch.int64, device="cuda")
    wire_len = torch.zeros(P, dtype=torch.int64, device="cuda")
    ctx.partition(st, part)
    ctx.pack(st, part, rec)

    def encode(**kw):
        ctx.delta_encode(rec, part.pair_off, None, None, ref, wire, wire_off, wire_len, **kw)

    def check():
        assert ctx.status(raise_on_error=False)[0] == tera.OK
        res = oracle.exchange_iteration(oracle.make_grid(wl.lo, wl.hi, wl.grid, wl.w), to_numpy(st))
        np.testing.assert_array_equal(wire_len.cpu().numpy().view(np.uint64), res["wire_len"])
        units = int(res["pair_off"][-1]) + P
        assert ref[:units * 64].cpu().numpy().tobytes() == res["ref_next"][:units * 64].tobytes()

    return ctx, encode, check


def captured_kernels(ctx, encode):
    ctx.profile(True)
    ctx.profile_table(reset=True)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        encode(stream=torch.cuda.current_stream())
    g.replay()
    torch.cuda.synchronize()
    names = set(ctx.profile_table(reset=True))
    ctx.profile(False)
    return names


def test_reserved_context_captures_the_encode_over_tiles():
    ctx, encode, check = encode_case(reserve=True)
    assert "codec_encode_kernel" in captured_kernels(ctx, encode)
    check()
    ctx.close()


def test_reserved_context_allocates_nothing_at_its_first_encode():
    ctx, encode, check = encode_case(reserve=True)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    encode()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == before
    check()
    ctx.close()


def test_captured_encode_without_the_scratch():
    ctx, encode, check = encode_case(reserve=False)
    encode(pair_begin=0, pair_end=27)  # the unit arrays, not the tiles' scratch
    names = captured_kernels(ctx, encode)
    assert "enc_emit_kernel" in names and "codec_encode_kernel" not in names
    check()
    encode()  # outside a capture the scratch is allocated
    check()
    assert "codec_encode_kernel" in captured_kernels(ctx, encode)
    check()
    ctx.close()


@pytest.mark.parametrize("eager,captured", [(None, (256, 4, 0, 0)), ((256, 4, 0, 0), None)])
def test_capture_of_the_other_form_of_the_batched_codec(eager, captured):
    import paper_2509_24063_gb300 as tera
    wl = Workload("t", 40000, (0.0,) * 3, (160.0,) * 3, (4, 4, 4), 12.0, 2, p_grow=0.1,
                  p_divide=0.02, p_die=0.02, seed=14)
    first, second = Generator(wl, device="cuda").series(2)
    g = oracle.make_grid(wl.lo, wl.hi, wl.grid, wl.w)
    res0 = oracle.exchange_iteration(g, to_numpy(first))
    res = oracle.exchange_iteration(g, to_numpy(second), ref=(res0["ref_next"], res0["pair_off"]),
                                    recv_ref=(res0["recv"], res0["recv_off"]))
    ctx = tera.Context(wl.lo, wl.hi, wl.grid, wl.w)
    ex = tera.AuraExchange(ctx, max_agents=60000, max_records=120000, path="batched", tune=eager)
    ex.step(first)
    ex.tune = captured
    graph = ex.capture(second)
    for _ in range(2):
        graph.replay()
    ex.advance()
    assert ctx.status(raise_on_error=False)[0] == tera.OK
    np.testing.assert_array_equal(ex.wire_len.cpu().numpy().view(np.uint64), res["wire_len"])
    units = int(res["pair_off"][-1]) + ctx.n_pairs
    for got, want in ((ex.sender_ref()[0], res["ref_next"]), (ex.receiver_ref()[0], res["recv"])):
        assert got[:units * 64].cpu().numpy().tobytes() == want[:units * 64].tobytes()
    ctx.close()


@pytest.mark.parametrize("tune", [None, (256, 4, 0, 0)])
def test_batched_exchange_is_captured_without_an_eager_step(tune):
    import paper_2509_24063_gb300 as tera
    wl = Workload("t", 40000, (0.0,) * 3, (160.0,) * 3, (4, 4, 4), 12.0, 1, seed=15)
    st = next(iter(Generator(wl, device="cuda").series(1)))
    ctx = tera.Context(wl.lo, wl.hi, wl.grid, wl.w)
    ex = tera.AuraExchange(ctx, max_agents=50000, max_records=120000, path="batched", tune=tune)
    graph = ex.capture(st)
    graph.replay()
    ex.advance()
    assert ctx.status(raise_on_error=False)[0] == tera.OK
    res = oracle.exchange_iteration(oracle.make_grid(wl.lo, wl.hi, wl.grid, wl.w), to_numpy(st))
    np.testing.assert_array_equal(ex.wire_len.cpu().numpy().view(np.uint64), res["wire_len"])
    units = int(res["pair_off"][-1]) + ctx.n_pairs
    for got, want in ((ex.sender_ref()[0], res["ref_next"]), (ex.receiver_ref()[0], res["recv"])):
        assert got[:units * 64].cpu().numpy().tobytes() == want[:units * 64].tobytes()
    ctx.close()
