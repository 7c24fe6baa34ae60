"""GPU: the ordered block products of Davidson against the shared ones of the matvec call, on
phase 1, where every sum is one task and both run the same loop: what keeps the order may not
cost FP64 operations of its own.  The limit of 1.5 lies between the two cases that can occur, no
further operation (1.0 to 1.1) and one multiplication per FMA (2.2), and the fastest of several
runs of each is compared, on a table that takes milliseconds."""
import pytest

from tests.test_gpu_parity import Context  # noqa: F401  (fixture)
from workloads import make_problem

pytestmark = pytest.mark.gpu


def test_phase1_ordered_against_shared(Context):  # noqa: F811
    import torch
    cfg, h, V = make_problem("random28")
    D, site = 700, cfg["L"] // 2 - 1
    ctx = Context(cfg["L"], cfg["group_irreps"], cfg["N"], cfg["two_S"], cfg["irrep"], group=7)
    ctx.set_integrals(h, V)
    ctx.set_schedule([D], [0.0], [1], [0.0], 1e-14, 3)
    ctx.init_mps(1)
    ctx.canonicalize(site)
    n, _ = ctx.layout(site)
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    y = torch.empty_like(x)

    def phase1(f):
        a = ctx.stats()
        f()
        b = ctx.stats()
        return (b["k_phase1_ms"] - a["k_phase1_ms"]) / (b["k_launches"] - a["k_launches"])
    shared = min(phase1(lambda: ctx.matvec(site, x, y)) for _ in range(5))
    ordered = min(phase1(lambda: ctx.davidson(site, x.clone())) for _ in range(4))
    assert ordered <= 1.5 * shared, (ordered, shared)
