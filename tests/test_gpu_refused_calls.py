"""A codec call refused for a wire that is too small changes nothing, and a raw
message that tera_reset_reference asked for is still raw on the retry, also when
the pair's message is empty; messages and totals against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from synth import to_numpy
from test_gpu_tiles import two_pairs

pytestmark = pytest.mark.gpu

FILL = 0xA5


@pytest.mark.parametrize("gone", [False, True])
@pytest.mark.parametrize("path", ["batched", "all_pairs"])
def test_reset_overflow_retry(path, gone):
    import paper_2509_24063_gb300 as tera
    first, second, _ = two_pairs(300, 200, 11)
    if gone:  # box 0's message is empty, while both sides' references hold its slots
        keep = ~((second["x"] >= 80) & (second["x"] < 100))
        second = {f: v[keep].contiguous() for f, v in second.items()}
    lo, hi, grid = (0.0,) * 3, (200.0, 100.0, 100.0), (2, 1, 1)
    g = oracle.make_grid(lo, hi, grid, 20.0)
    ctx = tera.Context(lo, hi, grid, 20.0)
    ex = tera.AuraExchange(ctx, max_agents=2000, max_records=4000, path=path)
    ex.step(first)
    ctx.status()
    res0 = oracle.exchange_iteration(g, to_numpy(first))
    res = oracle.exchange_iteration(g, to_numpy(second), ref=(res0["ref_next"], res0["pair_off"]),
                                    recv_ref=(res0["recv"], res0["recv_off"]))
    ex.part.pair_off = ex.pair_off[1]
    ctx.partition(second, ex.part)
    if path == "batched":
        ctx.pack_ids(second, ex.part, ex.rec, ex.rec_ids)
    else:
        ctx.pack(second, ex.part, ex.rec)
    ctx.status()
    for p in range(ctx.n_pairs):
        ctx.reset_reference(p)
    args, kw = ex.codec_args(1)

    def call(wire):
        a = list(args)
        a[5] = wire
        if path == "batched":
            ctx.codec_batched(*a, **kw)
        else:
            ctx.delta_encode(*a[:8])

    outputs = [ex.ref[1], ex.wire, ex.wire_len, ex.recv[1]]
    for t in outputs:
        t.view(torch.uint8).fill_(FILL)
    ctx.stats(reset=True)
    small = 64 * ctx.n_pairs  # every header fits, not every slab
    call(ex.wire[:small])
    code, req = ctx.status(raise_on_error=False)
    assert code == tera.ECAPACITY and req > small
    for t in outputs:
        assert bool((t.view(torch.uint8) == FILL).all())
    assert not any(ctx.stats().values())
    call(ex.wire[:req])
    if path != "batched":
        ctx.delta_decode(ex.wire, ex.wire_off, *args[8:])
    assert ctx.status(raise_on_error=False)[0] == tera.OK
    off = res["pair_off"]
    st, wire, wo, wl, nxt = oracle.encode_all(res["rec"], off, res0["ref_next"], res0["pair_off"],
                                              reset=np.ones(ctx.n_pairs, np.uint8))
    assert st == oracle.OK
    assert int(wo[-1]) == req
    got = ex.wire.cpu().numpy()
    np.testing.assert_array_equal(ex.wire_len.cpu().numpy().view(np.uint64), wl)
    for p in range(ctx.n_pairs):
        a, b = int(wo[p]), int(wo[p]) + int(wl[p])
        assert got[a:b].tobytes() == wire[a:b].tobytes(), p
        assert int(got[a + 12:a + 16].view(np.uint32)[0]) == oracle.MODE_RAW
    units = int(off[-1]) + ctx.n_pairs
    for arena in (ex.ref[1], ex.recv[1]):
        assert arena[:units * 64].cpu().numpy().tobytes() == nxt[:units * 64].tobytes()
    assert ctx.stats()["wire_bytes"] == int(wl.sum())
    ctx.close()


@pytest.mark.parametrize("a", [200, 5000])
@pytest.mark.parametrize("word", [0, 8, 12, 16])
def test_rejected_receiver_reference_skips_the_whole_pair(a, word):
    # a damaged header (magic, class, pair, count) of the receiver's reference, of a
    # pair of one and of several tiles; the persistent launch's receive buffer
    import paper_2509_24063_gb300 as tera
    first, second, _ = two_pairs(a, 300, 3)
    lo, hi, grid = (0.0,) * 3, (200.0, 100.0, 100.0), (2, 1, 1)
    buffers = []
    for tune in (None, (256, 4, 0, 0)):
        ctx = tera.Context(lo, hi, grid, 20.0)
        ex = tera.AuraExchange(ctx, max_agents=12000, max_records=30000, path="batched", tune=tune)
        ex.step(first)
        ctx.status()
        off = ex.recv_off[0].cpu().numpy()
        p = int(np.argmax(off[1:] - off[:-1] == a))
        assert off[p + 1] - off[p] == a
        ex.recv[0][(int(off[p]) + p) * 64 + word] ^= 1
        ex.recv[1].zero_()
        ex.step(second)
        code, _ = ctx.status(raise_on_error=False)
        assert code == tera.ECORRUPT
        off = ex.recv_off[1].cpu().numpy()
        units = int(off[-1]) + ctx.n_pairs
        got = ex.recv[1][:units * 64].cpu().numpy()
        assert not got[(int(off[p]) + p + 1) * 64:(int(off[p + 1]) + p + 1) * 64].any()
        buffers.append(got.tobytes())
        ctx.close()
    assert buffers[0] == buffers[1]
