"""The codec over tiles (batched without an explicit schedule, and the encode
of every pair) at the sizes where its
steps, tiles and ways of matching change, byte for byte against the oracle."""
import numpy as np
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


def run_states(tera, states, lo, hi, grid, w, id_columns=True, path="batched"):
    ctx = tera.Context(lo, hi, grid, w)
    nmax = max(int(s["x"].shape[0]) for s in states)
    ex = tera.AuraExchange(ctx, max_agents=nmax, max_records=3 * nmax + 1024, path=path,
                           id_columns=id_columns)
    g = oracle.make_grid(lo, hi, grid, w)
    ref = recv_ref = None
    for st in states:
        ex.step(st)
        code, _ = ctx.status(raise_on_error=False)
        assert code == tera.OK
        res = oracle.exchange_iteration(g, to_numpy(st), ref=ref, recv_ref=recv_ref)
        compare_iteration(ctx, ex, st, res, ctx.n_pairs)
        ref, recv_ref = (res["ref_next"], res["pair_off"]), (res["recv"], res["recv_off"])
    ctx.close()


def two_pairs(a, b, seed):
    """Three states of two boxes (2 x 1 x 1) whose two messages start with a and
    b records: in the second some agents are gone, some new and some moved; in
    the third every agent has another id, so nothing matches."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n = a + b + 40

    def rand(k):
        return torch.rand(k, generator=g, device="cuda", dtype=torch.float64)

    def state(ids):
        k = ids.numel()
        return dict(id=ids, x=torch.empty(k, device="cuda", dtype=torch.float64), y=100 * rand(k),
                    z=100 * rand(k), diameter=8 + 4 * rand(k), volume=rand(k),
                    adherence=rand(k), density=torch.ones(k, device="cuda", dtype=torch.float64))

    st = state(torch.arange(n, device="cuda"))
    # box 0 is [0, 100), box 1 [100, 200), the aura 20 wide
    st["x"][:a] = 80 + 20 * rand(a)
    st["x"][a:a + b] = 100 + 20 * rand(b)
    st["x"][a + b:] = 5 + 20 * rand(40)
    keep = rand(n) >= 0.1
    second = {f: v[keep].clone() for f, v in st.items()}
    k = second["x"].shape[0]
    move = rand(k) < 0.3
    second["y"] = torch.where(move, second["y"] * 0.999, second["y"])
    new = max(1, n // 15)
    born = state(torch.arange(n, n + new, device="cuda"))
    born["x"][:] = 80 + 40 * rand(new)
    second = {f: torch.cat([v, born[f]]) for f, v in second.items()}
    third = {f: v.clone() for f, v in second.items()}
    third["id"] = third["id"] + 10 * n
    return [st, second, third]


@pytest.mark.parametrize("path", ["batched", "all_pairs"])
@pytest.mark.parametrize("order", ["ascending", "shuffled"])
@pytest.mark.parametrize("a,b", [(0, 0), (1, 0), (31, 33), (32, 64), (63, 65), (255, 257),
                                 (511, 513), (3136, 3137), (2047, 4097), (6272, 6273), (8191, 8192),
                                 (8193, 70000)])
def test_pair_sizes_at_the_edges(tera, a, b, order, path):
    states = two_pairs(a, b, 7 * a + b)
    if order == "shuffled":  # a message's ids in no order: the hash tables match them
        g = torch.Generator(device="cuda")
        g.manual_seed(a + b)
        for k, st in enumerate(states):
            perm = torch.randperm(st["x"].shape[0], generator=g, device="cuda")
            states[k] = {f: v[perm].contiguous() for f, v in st.items()}
    run_states(tera, states, (0.0,) * 3, (200.0, 100.0, 100.0), (2, 1, 1), 20.0, path=path)


@pytest.mark.parametrize("id_columns", [True, False])
@pytest.mark.parametrize("shuffle", [False, True])
def test_small_pairs_of_a_large_grid(tera, shuffle, id_columns):
    # 13,824 pairs, most of them small or empty: matched a warp each
    wl = Workload("t", 120000, (0.0,) * 3, (400.0, 400.0, 400.0), (8, 8, 8), 15.0, 4,
                  p_grow=0.1, p_divide=0.02, p_die=0.02, seed=77)
    states = [{f: v for f, v in st.items()} for st in Generator(wl, device="cuda").series(4)]
    if shuffle:
        states = [{f: v.flip(0).contiguous() for f, v in st.items()} for st in states]
    run_states(tera, states, wl.lo, wl.hi, wl.grid, wl.w, id_columns=id_columns)


def test_reset_pairs_are_sent_raw(tera):
    # half of the pairs marked for a raw message in the middle of a chain, in
    # both directions of a pair
    states = two_pairs(700, 9000, 5)[:2]
    lo, hi, grid = (0.0,) * 3, (200.0, 100.0, 100.0), (2, 1, 1)
    ctx = tera.Context(lo, hi, grid, 20.0)
    ex = tera.AuraExchange(ctx, max_agents=12000, max_records=30000, path="batched")
    g = oracle.make_grid(lo, hi, grid, 20.0)
    ex.step(states[0])
    res0 = oracle.exchange_iteration(g, to_numpy(states[0]))
    reset = np.zeros(ctx.n_pairs, np.uint8)
    for p in range(0, ctx.n_pairs, 2):
        ctx.reset_reference(p)
        reset[p] = 1
    ex.step(states[1])
    ctx.status()
    res = oracle.exchange_iteration(g, to_numpy(states[1]), ref=(res0["ref_next"], res0["pair_off"]),
                                    recv_ref=(res0["recv"], res0["recv_off"]))
    off = res["pair_off"]
    st, wire, wo, wl, nxt = oracle.encode_all(res["rec"], off, res0["ref_next"], res0["pair_off"],
                                              reset=reset)
    assert st == oracle.OK
    got = ex.wire.cpu().numpy()
    np.testing.assert_array_equal(ex.wire_len.cpu().numpy().view(np.uint64), wl)
    for p in range(ctx.n_pairs):
        a, b = int(wo[p]), int(wo[p]) + int(wl[p])
        assert got[a:b].tobytes() == wire[a:b].tobytes(), p
    units = int(off[-1]) + ctx.n_pairs
    for arena in (ex.sender_ref()[0], ex.receiver_ref()[0]):
        assert arena[:units * 64].cpu().numpy().tobytes() == nxt[:units * 64].tobytes()
    ctx.close()
