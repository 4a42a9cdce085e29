"""The work that users of this framework have it do, as cases that can be timed.

A case is one pass through the public entry points: one aura-exchange
iteration (eager or replayed from a CUDA graph, batched or call by call, plain
or with the learned predictor), one migration step, one training run of the
predictor, or one exchange step on host-resident state.  Populations follow
the repository's workloads: uniform or blob layouts, agents that move, grow,
divide and die between two iterations, closed or toroidal domains.

The message of iteration 0 is every pass's reference: the exchanges are made
with a reference interval that never ends (or replay the graph of one
iteration), so that a pass repeats one and the same iteration of a chain.
"""
import math

import numpy as np
import torch

import paper_2509_24063_gb300 as tera
from paper_2509_24063_gb300.host import HostExchange
from paper_2509_24063_gb300.migrate import Migration

FIELDS = ("id", "x", "y", "z", "diameter", "volume", "adherence", "density")
AXES = ("x", "y", "z")
FOREVER = 1 << 30  # reference interval: iteration 0 stays the reference

# 8 -> 64 -> 64 -> 3 network of the predictor: offsets of its seven parts
W1, B1, W2, B2, W3, B3, PARAMS = 0, 512, 576, 4672, 4736, 4928, 4931


# ---------------- the cases ----------------

def _step(name, agents, grid, side, w, **kw):
    """One exchange iteration; `side` is a box's side, `w` the aura width."""
    c = dict(kind="step", agents=agents, gx=grid[0], gy=grid[1], gz=grid[2], side=float(side),
             w=float(w), layout="uniform", periodic=0, order="id", path="batched", graph=False,
             divide=0.005, die=0.002)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest simulation: a few thousand cells in four boxes, stepped
        # eagerly; launches and host work are all there is
        _step("step_4k", 4096, (2, 2, 1), 50, 30, divide=0.0, die=0.0),
        # a small, odd population on a ragged box grid, its iteration replayed
        # from a CUDA graph as an inner loop does
        _step("step_100k_ragged", 99991, (5, 3, 2), 100, 25, graph=True),
        # an ordinary simulation of a million cells, stepped eagerly
        _step("step_1m", 1 << 20, (4, 4, 4), 250, 30),
        # the same on a toroidal domain through the separate pack, encode and
        # decode calls, which ranks that exchange messages use
        _step("calls_1m_torus", 1 << 20, (4, 4, 4), 250, 30, path="all_pairs", periodic=7),
        # clustered tissue: box loads that differ by a factor of ten
        _step("step_16m_blobs", 16 << 20, (4, 4, 4), 1000, 30, layout="blobs"),
        # a simulation whose agents migrate: the state is kept box by box, so a
        # message's ids are in no order
        _step("step_16m_migrated", 16 << 20, (8, 8, 8), 500, 30, order="box", divide=0.0, die=0.0),
        # the largest population of one GPU, replayed from a graph
        _step("step_100m", 100_000_000, (8, 8, 8), 1000, 30, graph=True, divide=0.01, die=0.01),
        # drifting blob agents with the learned predictor's residual messages
        dict(name="predict_16m", kind="predict", agents=16 << 20, gx=4, gy=4, gz=4, side=1000.0,
             w=30.0, layout="blobs"),
        # a hundred steps of the predictor's training at its default batch
        dict(name="train_8k", kind="train", samples=1 << 20, batch=8192, steps=100),
        # migration between the boxes of an ordinary and of the largest population
        dict(name="migrate_1m", kind="migrate", agents=1 << 20, gx=4, gy=4, gz=4, side=250.0,
             w=30.0, periodic=0, sigma=0.5),
        dict(name="migrate_100m", kind="migrate", agents=100_000_000, gx=8, gy=8, gz=8,
             side=1000.0, w=30.0, periodic=0, sigma=0.5),
        # a simulation on the host that hands over its state and takes the
        # iteration's messages back
        dict(name="host_1m", kind="host", agents=1 << 20, gx=4, gy=4, gz=4, side=250.0, w=30.0),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _grid(rng):
    return tuple(int(round(_log(rng, 1, 8))) for _ in range(3))


def _capped(agents, c):
    """Fewer agents where wide auras would make the case dearer than the largest."""
    ratio = _entry_ratio(c)
    return max(1000, min(agents, int(90_000_000 / (1.0 + 21.0 * ratio) * 4.4)))


def draw(rng):
    kind = rng.choice(("step",) * 5 + ("calls", "predict", "train", "migrate", "host"))
    if kind == "train":
        batch = int(_log(rng, 200, 32768))
        return dict(kind="train", samples=int(_log(rng, 20_000, 2_000_000)), batch=batch,
                    steps=max(10, min(200, 1_000_000 // batch)))
    grid = _grid(rng)
    if grid == (1, 1, 1):
        grid = (2, 1, 1)
    side = _log(rng, 50, 1000)
    c = dict(gx=grid[0], gy=grid[1], gz=grid[2], side=side, w=side * _log(rng, 0.02, 0.6))
    if kind == "predict":
        agents = int(_log(rng, 20_000, 8_000_000))
        return dict(kind="predict", agents=_capped(agents, dict(c, periodic=0)) // 2,
                    layout=rng.choice(("uniform", "blobs")), **c)
    if kind == "host":
        return dict(kind="host", agents=int(_log(rng, 4_000, 2_000_000)), **c)
    periodic = 0
    if rng.random() < 0.3:
        periodic = sum(1 << a for a in range(3) if grid[a] >= 3)
    if kind == "migrate":
        return dict(kind="migrate", agents=int(_log(rng, 4_000, 64_000_000)), periodic=periodic,
                    sigma=0.5, **c)
    agents = int(_log(rng, 2_000, 64_000_000 if kind == "step" else 4_000_000))
    grow = rng.random() < 0.7
    order = rng.choice(("id", "id", "box"))
    return dict(kind="step", agents=_capped(agents, dict(c, periodic=periodic)),
                layout=rng.choice(("uniform", "uniform", "blobs")), periodic=periodic, order=order,
                path="batched" if kind == "step" else "all_pairs", graph=rng.random() < 0.5,
                divide=0.005 if grow and order == "id" else 0.0,
                die=0.002 if grow and order == "id" else 0.0, **c)


# ---------------- populations ----------------

class _Population:
    """Seeded agents on the GPU and the operations between two iterations."""

    def __init__(self, case, seed):
        self.dev = torch.device("cuda")
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(int(seed))
        self.rng = np.random.default_rng(int(seed))
        self.n = (case["gx"], case["gy"], case["gz"])
        self.side, self.w = case["side"], case["w"]
        self.hi = tuple(k * self.side for k in self.n)
        self.periodic = case.get("periodic", 0)
        self.layout = case.get("layout", "uniform")
        self.agents = self.next_id = int(case["agents"])
        # capacities a user provisions: for the births of an iteration, and for
        # the expected aura records with a margin (blobs: several times that)
        births = case.get("divide", 0.0) * self.agents
        self.max_agents = int(self.agents + births + 8.0 * math.sqrt(births)) + 64
        margin = 4.0 if self.layout == "blobs" else 1.1
        self.max_records = int(margin * _entry_ratio(case) * self.max_agents) + 4096

    def context(self):
        return tera.Context((0.0, 0.0, 0.0), self.hi, self.n, self.w, periodic=self.periodic)

    def rand(self, n):
        return torch.rand(n, generator=self.g, device=self.dev, dtype=torch.float64)

    def randn(self, n):
        return torch.randn(n, generator=self.g, device=self.dev, dtype=torch.float64)

    def bound(self, a, v):
        hi = self.hi[a]
        if self.periodic >> a & 1:
            v = torch.remainder(v, hi)
        return v.clamp_(0.0, math.nextafter(hi, 0.0))

    def initial(self):
        """The agents of iteration 0 (blobs that would come near the records'
        capacity are drawn again)."""
        for _ in range(64):
            st = self._initial()
            if self.layout != "blobs" or self.entries(st) < 0.9 * self.max_records:
                return st
        raise RuntimeError("no blobs that fit the records' capacity")

    def _initial(self):
        n = self.agents
        if self.layout == "blobs":
            size = max(self.hi)
            sigma = self.rng.uniform(0.005, 0.05, 32) * size
            share = torch.tensor(self.rng.dirichlet(np.full(32, 0.5)), device=self.dev)
            centre = self.rng.uniform(np.zeros(3), np.array(self.hi), (32, 3))
            blob = torch.searchsorted(share.cumsum(0), self.rand(n)).clamp_(max=31)
            sig = torch.tensor(sigma, device=self.dev)[blob]
            ctr = torch.tensor(centre, device=self.dev)[blob]
            pos = [self.bound(a, ctr[:, a] + sig * self.randn(n)) for a in range(3)]
        else:
            pos = [self.bound(a, self.hi[a] * self.rand(n)) for a in range(3)]
        d = 8.0 + 4.0 * self.rand(n)
        return dict(id=torch.arange(n, device=self.dev), x=pos[0], y=pos[1], z=pos[2], diameter=d,
                    volume=(math.pi / 6.0) * d * d * d, adherence=0.3 + 0.4 * self.rand(n),
                    density=torch.ones(n, device=self.dev, dtype=torch.float64))

    def move(self, st, sigma=0.5):
        n = st["x"].shape[0]
        mv = self.rand(n) < 0.3
        st = {k: v.clone() for k, v in st.items()}
        for a, k in enumerate(AXES):
            st[k] = self.bound(a, torch.where(mv, st[k] + sigma * self.randn(n), st[k]))
        return st

    def live(self, st, divide, die):
        """Moves; a tenth of the agents grow; some divide, some die."""
        st = self.move(st)
        n = st["x"].shape[0]
        d = torch.where(self.rand(n) < 0.1, st["diameter"] * 1.01, st["diameter"])
        st["diameter"], st["volume"] = d, (math.pi / 6.0) * d * d * d
        if divide > 0:
            dv = torch.nonzero(self.rand(n) < divide).flatten()
            k = dv.numel()
            u = torch.stack([self.randn(k) for _ in range(3)], 1)
            u = u / u.norm(dim=1, keepdim=True).clamp_min(1e-300)
            child = {f: v[dv] for f, v in st.items()}
            small = child["diameter"] * 2.0 ** (-1.0 / 3.0)
            for a, ax in enumerate(AXES):
                child[ax] = self.bound(a, child[ax] + 0.5 * child["diameter"] * u[:, a])
            child["diameter"] = small
            child["volume"] = (math.pi / 6.0) * small * small * small
            st["diameter"][dv], st["volume"][dv] = child["diameter"], child["volume"]
            child["id"] = torch.arange(self.next_id, self.next_id + k, device=self.dev)
            self.next_id += k
            st = {f: torch.cat([v, child[f]]) for f, v in st.items()}
        if die > 0:
            keep = self.rand(st["x"].shape[0]) >= die
            st = {f: v[keep] for f, v in st.items()}
        return st

    def drift(self, st, vel):
        """Persistent motion: a tenth of each velocity is renewed by noise."""
        n = st["x"].shape[0]
        st = {k: v.clone() for k, v in st.items()}
        for a, k in enumerate(AXES):
            vel[a] = 0.8 * vel[a] + 0.02 * self.randn(n) + 0.1 * torch.sin(st[AXES[a - 1]] / 500.0)
            st[k] = self.bound(a, st[k] + vel[a])
        return st

    def entries(self, st):
        """Aura records of a state: over the axes, the product of one and the
        number of neighbours whose aura holds the coordinate, less the agent."""
        prod = None
        for a, ax in enumerate(AXES):
            v, n = st[ax], self.n[a]
            box = (v / self.side).floor_().clamp_(0, n - 1)
            per = bool(self.periodic >> a & 1)
            k = 1 + ((v < box * self.side + self.w) & ((box > 0) | per)).to(torch.int32)
            k += (v >= (box + 1) * self.side - self.w) & ((box < n - 1) | per)
            prod = k if prod is None else prod * k
        return int(prod.sum()) - st["x"].shape[0]


def _migrated(pop, ctx, st, box_off):
    """A box-major state moved and regrouped, as a simulation does between two exchanges."""
    mig = Migration(ctx, pop.agents, max_leavers=pop.agents)
    if box_off is None:
        return mig.regroup(st)
    return mig.step(pop.move(st), box_off)


def _blank(ex):
    """Zeroes in the buffers the next iteration writes: the parts of a buffer that
    no message occupies then hold the same bytes at every pass."""
    for t in (ex.part.owner, ex.part.mask, ex.part.pair_idx, ex.rec, ex.ref[1], ex.recv[1], ex.wire):
        t.zero_()


# ---------------- prepare and run ----------------

def prepare(case, seed):
    return {"step": _prepare_step, "predict": _prepare_predict, "train": _prepare_train,
            "migrate": _prepare_migrate, "host": _prepare_host}[case["kind"]](case, seed)


def run(state):
    return state["run"](state)


def _outputs(ex, more=()):
    out = dict(owner=ex.part.owner, mask=ex.part.mask, pair_count=ex.part.pair_count,
               pair_off=ex.pair_off[1], pair_idx=ex.part.pair_idx, messages=ex.rec, wire=ex.wire,
               wire_off=ex.wire_off, wire_len=ex.wire_len, sender_ref=ex.ref[1],
               receiver_ref=ex.recv[1], receiver_off=ex.recv_off[1])
    out.update(more)
    return out


def _run_step(s):
    s["ex"].step(s["agents"])
    return _outputs(s["ex"])


def _run_graph(s):
    s["graph"].replay()
    s["ex"].advance()
    return _outputs(s["ex"], s.get("more", ()))


def _prepare_step(case, seed):
    pop = _Population(case, seed)
    ctx = pop.context()
    a = pop.initial()
    if case["order"] == "box":
        a, off = _migrated(pop, ctx, a, None)
        b, _ = _migrated(pop, ctx, a, off)
    else:
        b = pop.live(a, case["divide"], case["die"])
    ex = tera.AuraExchange(ctx, pop.max_agents, pop.max_records, path=case["path"],
                           ref_interval=FOREVER)
    ex.step(a)
    ctx.status()
    _blank(ex)
    s = dict(run=_run_step, ctx=ctx, ex=ex, agents=b)
    if case["graph"]:
        s.update(run=_run_graph, graph=ex.capture(b))
    return s


def _network():
    """A network that expects four fifths of the last displacement, its other
    weights small: what training on such motion arrives at."""
    p = torch.zeros(PARAMS)
    g = torch.Generator()
    g.manual_seed(1)
    p[W1:B1] = 1e-6 * torch.randn(512, generator=g)
    p[W2:B2] = 1e-6 * torch.randn(4096, generator=g)
    for a in range(3):
        for h, sign in ((2 * a, 1.0), (2 * a + 1, -1.0)):
            p[W1 + 8 * h + a] = sign
            p[W2 + 64 * h + h] = 1.0
            p[W3 + 64 * a + h] = 0.8 * sign
    return p.cuda()


def _prepare_predict(case, seed):
    pop = _Population(case, seed)
    ctx = pop.context()
    states, vel = [pop.initial()], [0.0, 0.0, 0.0]
    for _ in range(3):
        states.append(pop.drift(states[-1], vel))
    # three iterations give the references the two displacements a prediction
    # needs; the graph is that of the fourth
    ex = tera.AuraExchange(ctx, pop.max_agents, pop.max_records, path="batched",
                           params=_network())
    for st in states[:3]:
        ex.step(st)
    ctx.status()
    _blank(ex)
    for h in (ex.hist[1], ex.rhist[1]):
        h.zero_()
    more = dict(sender_history=ex.hist[1], receiver_history=ex.rhist[1])
    return dict(run=_run_graph, ctx=ctx, ex=ex, agents=states[3], graph=ex.capture(states[3], t=3),
                more=more)


def _train_inputs(case, seed):
    """Samples as the encoder writes them: two displacements, a diameter, a
    neighbour count, the next displacement; one in ten rows is not valid."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    n = case["samples"]
    d1 = 0.5 * torch.randn(n, 3, generator=g, device="cuda")
    d2 = 0.8 * d1 + 0.3 * torch.randn(n, 3, generator=g, device="cuda")
    s = torch.empty(n, 12, device="cuda")
    s[:, 0:3], s[:, 3:6] = d1, d2
    s[:, 6] = 0.8 + 0.4 * torch.rand(n, generator=g, device="cuda")
    s[:, 7] = torch.randint(1, 40, (n,), generator=g, device="cuda") / 32.0
    s[:, 8:11] = 0.8 * d1 + 0.1 * torch.randn(n, 3, generator=g, device="cuda")
    s[:, 11] = (torch.rand(n, generator=g, device="cuda") < 0.9).float()
    p = torch.zeros(PARAMS, device="cuda")
    for o, fan_in, fan_out in ((W1, 8, 64), (W2, 64, 64), (W3, 64, 3)):
        u = torch.rand(fan_in * fan_out, generator=g, device="cuda") * 2 - 1
        p[o:o + u.numel()] = u * math.sqrt(6.0 / fan_in) * (0.1 if fan_out == 3 else 1.0)
    return s.reshape(-1), p


LR, CLIP = 0.02, 1.0


def _prepare_train(case, seed):
    samples, params = _train_inputs(case, seed)
    small = tera.Context((0.0, 0.0, 0.0), (100.0, 100.0, 50.0), (2, 2, 1), 30.0)
    return dict(run=_run_train, ctx=small, samples=samples, params=params, case=case)


def _run_train(s):
    p = s["params"].clone()
    valid = s["ctx"].mlp_train(s["samples"], p, s["case"]["steps"], s["case"]["batch"], LR, CLIP)
    return dict(params=p, valid=valid)


def _prepare_migrate(case, seed):
    pop = _Population(case, seed)
    ctx = pop.context()
    st, off = _migrated(pop, ctx, pop.initial(), None)
    prev = pop.move(st, case["sigma"])
    mig = Migration(ctx, pop.agents)
    nxt = {k: torch.zeros_like(v) for k, v in prev.items()}
    return dict(run=_run_migrate, ctx=ctx, mig=mig, prev=prev, off=off, next=nxt,
                next_off=torch.zeros_like(off))


def _run_migrate(s):
    st, off = s["mig"].step(s["prev"], s["off"], s["next"], s["next_off"])
    # records are moved, not computed: their columns as the bits they are
    bits = {k: v.view(torch.int64) for k, v in st.items()}
    return dict(bits, box_off=off, inbox_off=s["mig"].inbox_off, inboxes=s["mig"].arena)


def _prepare_host(case, seed):
    pop = _Population(dict(case, divide=0.005), seed)
    ctx = pop.context()
    a = pop.initial()
    b = pop.live(a, 0.005, 0.002)
    hx = HostExchange(ctx, pop.max_agents, pop.max_records, ref_interval=FOREVER)
    out = torch.zeros(hx.wire_capacity, dtype=torch.uint8).pin_memory()
    hx.step({f: a[f].cpu().pin_memory() for f in FIELDS}, out).wait()
    ctx.status()
    _blank(hx.ex)
    out.zero_()
    return dict(run=_run_host, ctx=ctx, hx=hx, agents={f: b[f].cpu().pin_memory() for f in FIELDS},
                out=out)


def _run_host(s):
    n = s["hx"].step(s["agents"], s["out"]).wait()
    return dict(wire=s["out"], bytes=n)


# ---------------- what a pass cannot do without ----------------

def _entry_ratio(c):
    """Aura records per agent of a uniform population (blobs come near it)."""
    prod = 1.0
    for a, n in enumerate((c["gx"], c["gy"], c["gz"])):
        strips = 2 * n if c.get("periodic", 0) >> a & 1 else 2 * (n - 1)
        prod *= 1.0 + strips * c["w"] / (n * c["side"])
    return prod - 1.0


def _in_aura(c):
    """Share of the agents that are in some aura."""
    inside = 1.0
    for a, n in enumerate((c["gx"], c["gy"], c["gz"])):
        strips = 2 * n if c.get("periodic", 0) >> a & 1 else 2 * (n - 1)
        inside *= max(0.0, 1.0 - strips * c["w"] / (n * c["side"]))
    return 1.0 - inside


def work(case):
    if case["kind"] == "train":
        # the valid rows of the samples; forward, and backward to every weight
        # and to the first layer's activations
        mults = 512 + 4096 + 192
        per = 2 * (2 * mults + 4096 + 192)
        return {"bytes": 48 * case["samples"] + 8 * PARAMS,
                "flops": per * case["batch"] * case["steps"]}
    n = case["agents"]
    if case["kind"] == "migrate":
        # every agent's eight columns read and written
        return {"bytes": 128 * n, "flops": 0}
    e = _entry_ratio(case) * n
    # positions of all agents, the other columns of those in an aura; owner and
    # mask; per record: list entry, message, both new references written, both
    # references read, about 12 bytes of wire
    b = 24 * n + 40 * _in_aura(case) * n + 8 * n + (4 + 3 * 64 + 2 * 64 + 12) * e
    flops = 0
    if case["kind"] == "predict":
        b += 4 * 48 * e  # the histories of both sides, read and written
        flops = 2 * 2 * 4800 * e
    if case["kind"] == "host":
        b += 64 * n + 12 * e
    return {"bytes": b, "flops": flops}


# ---------------- 64-bit values ----------------

def exact(case, seed):
    """The trained weights in binary64; every other output is bytes or whole numbers."""
    if case["kind"] != "train":
        return None
    samples, params = _train_inputs(case, seed)
    rows = samples.reshape(-1, 12)
    rows = rows[rows[:, 11] != 0].double()
    f, y, nv, batch = rows[:, 0:8], rows[:, 8:11], rows.shape[0], case["batch"]
    p = params.double()
    lr = float(np.float32(LR))
    for k in range(case["steps"]):
        at = (torch.arange(batch, device=p.device) + (k * batch) % nv) % nv
        x, t = f[at], y[at]
        w1, w2, w3 = p[W1:B1].view(64, 8), p[W2:B2].view(64, 64), p[W3:B3].view(3, 64)
        a1 = (x @ w1.t() + p[B1:W2]).relu()
        a2 = (a1 @ w2.t() + p[B2:W3]).relu()
        go = 2.0 * (a2 @ w3.t() + p[B3:] - t) / batch
        g2 = (go @ w3) * (a2 > 0)
        g1 = (g2 @ w2) * (a1 > 0)
        grad = torch.cat([(g1.t() @ x).flatten(), g1.sum(0), (g2.t() @ a1).flatten(), g2.sum(0),
                          (go.t() @ a2).flatten(), go.sum(0)])
        norm = float(grad.norm())
        p = p - lr * (CLIP / norm if norm > CLIP else 1.0) * grad
    return dict(params=p, valid=None)
