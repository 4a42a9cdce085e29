"""An exchange step whose columns other than the positions arrive late, on
another stream, gives the bytes of a step on the whole state."""
import pytest
import torch

from test_gpu_host import FIELDS, workload
from synth import Generator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 4099])
@pytest.mark.parametrize("path", ["batched", "all_pairs", "per_subdomain"])
def test_late_columns(n, path):
    import paper_2509_24063_gb300 as tera
    wl = workload(n=4099, iters=1, seed=79)
    st = {f: v[:n].cuda() for f, v in next(iter(Generator(wl, device="cpu").series(1))).items()
          if f in FIELDS}
    outs = []
    for late in (False, True):
        ctx = tera.Context(wl.lo, wl.hi, wl.grid, wl.w)
        ex = tera.AuraExchange(ctx, 5000, 40000, path=path)
        ex.step(st)  # workspaces in place, and a reference for the next step
        ex.wire.zero_()  # what lies between two messages is not written
        view = {f: torch.zeros_like(v) for f, v in st.items()} if late else st
        torch.cuda.synchronize()
        if late:
            side = torch.cuda.Stream()
            with torch.cuda.stream(side):
                for f in ("x", "y", "z"):
                    view[f].copy_(st[f])
                there = torch.cuda.Event()
                there.record()
                torch.cuda._sleep(20_000_000)  # about 10 ms
                for f in FIELDS:
                    view[f].copy_(st[f])
                ready = torch.cuda.Event()
                ready.record()
            torch.cuda.current_stream().wait_event(there)
            ex.step(view, columns_ready=ready)
        else:
            ex.step(view)
        ctx.status()
        end = int(ex.wire_off[-1])
        outs.append((ex.wire_off.clone(), ex.wire[:end].clone()))
        ctx.close()
    assert torch.equal(outs[0][0], outs[1][0])
    assert torch.equal(outs[0][1], outs[1][1])
