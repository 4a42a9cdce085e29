"""The partition and its sort where their work is cut finer: at the edges of
the finer tiles and on both sides of each line between the two cuts, byte for
byte against the oracle."""
import pytest
import torch

from synth import Generator, Workload
from test_gpu_partition_sizes import one_iteration

pytestmark = pytest.mark.gpu


def line():
    """Agents from which the agent passes take four rounds a block."""
    return torch.cuda.get_device_properties(0).multi_processor_count * 4 * 2048


@pytest.mark.parametrize("entries", [1023, 1024, 1025, 307_200, 307_201])
def test_sort_tiles(entries):
    import paper_2509_24063_gb300 as tera
    g = torch.Generator(device="cuda")
    g.manual_seed(entries)

    def rand():
        return torch.rand(entries, generator=g, device="cuda", dtype=torch.float64)

    st = dict(id=torch.arange(entries, device="cuda"), x=85 + 30 * rand(), y=100 * rand(),
              z=100 * rand(), diameter=rand(), volume=rand(), adherence=rand(), density=rand())
    assert one_iteration(tera, st, (0.0,) * 3, (200.0, 100.0, 100.0), (2, 1, 1), 20.0,
                         entries + 7) == entries


@pytest.mark.parametrize("n", [511, 513, 1025, -1, 0])  # the last two: beside the line
def test_agent_rounds(n):
    import paper_2509_24063_gb300 as tera
    n = n if n > 0 else line() + n
    wl = Workload("t", n, (0.0,) * 3, (200.0, 150.0, 100.0), (4, 3, 2), 1.0, 1, seed=n)
    st = next(iter(Generator(wl, device="cuda").series(1)))
    one_iteration(tera, st, wl.lo, wl.hi, wl.grid, wl.w, n + 1024)
