"""GPU: which kernel sums the ordered block products of large blocks.  The kernel in rounds is for
tables too small to fill the SMs; on blocks of up to 90 rows with lists of hundreds of tasks it
runs at half the rate of the lanes.  Phase 2 of Davidson's products against the matvec call's
shared sums of the same table: 1.1 in lanes, 2.4 in rounds, and the limit of 1.6 in between; the
fastest of several runs of each, tens of milliseconds long."""
import pytest

from tests.test_gpu_parity import Context  # noqa: F401  (fixture)
from workloads import hubbard_chain

pytestmark = pytest.mark.gpu


def test_phase2_ordered_against_shared(Context):  # noqa: F811
    import torch
    L, D = 16, 1000
    ctx = Context(L, [0] * L, L, 0, 0)
    ctx.set_integrals(*hubbard_chain(L, 1.0, 4.0))
    ctx.set_schedule([D], [0.0], [1], [0.0], 1e-14, 3)
    ctx.init_mps(1)
    site = L // 2 - 1
    ctx.canonicalize(site)
    ctx.sweep_step(site, 1, D)
    site += 1
    n, _ = ctx.layout(site)
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    y = torch.empty_like(x)

    def phase2(f):
        a = ctx.stats()
        f()
        b = ctx.stats()
        return (b["k_phase2_ms"] - a["k_phase2_ms"]) / (b["k_launches"] - a["k_launches"])
    shared = min(phase2(lambda: ctx.matvec(site, x, y)) for _ in range(5))
    ordered = min(phase2(lambda: ctx.davidson(site, x.clone())) for _ in range(4))
    assert ordered <= 1.6 * shared, (ordered, shared)
