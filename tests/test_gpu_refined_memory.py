"""GPU: dmrg_truncate under device-memory caps.  The refined eigensolver needs more than the
Jacobi solver in place, which takes over wherever an allocation of the first fails: as the cap
rises, calls fail, then succeed in place, then refined, with nothing refused in between.  A call
that fails leaves no device bytes behind, one that succeeds gives the same state.

Tolerances: both solvers have eigenvalue errors of ~1e-15 of the largest, 1e-12 is asked of the
discarded weight; the cut is placed at a gap, so the states agree to ~1e-13, 1e-10 is asked."""
import numpy as np
import pytest

from tests.test_gpu_parity import Context  # noqa: F401  (fixture)
from tests.test_gpu_refined_decomposition import vector
from workloads import hubbard_chain

pytestmark = pytest.mark.gpu


# sectors of at most 64 rows, and above (block Jacobi, whose buffers come last)
@pytest.mark.parametrize("L,D,caps", [(12, 400, 160), (12, 1500, 80)])
@pytest.mark.parametrize("direction", [1, -1])
def test_caps_refuse_nothing_that_fits_in_place(Context, L, D, caps, direction):  # noqa: F811
    from paper_1312_2415_gb300 import binding
    site = L // 2 - 1
    ctx = Context(L, [0] * L, L, 0, 0)
    ctx.set_integrals(*hubbard_chain(L, 1.0, 4.0))
    ctx.set_schedule([D], [1e-8], [1], [0.0])
    ctx.init_mps(3)
    ctx.canonicalize(site)
    x = vector(ctx, site, "falling", 5)

    def launches(f):
        a = ctx.stats()["kernels_launched"]
        out = f()
        return out, ctx.stats()["kernels_launched"] - a

    w, refined = launches(lambda: ctx.truncate(site, direction, D // 2, x))
    y = ctx.tt_to_x(site)
    used = binding.device_memory_in_use()
    n = ctx.layout(site)[0]
    count, refused, served = [], [], []
    try:
        for room in 8 * n * np.geomspace(1.0, 64.0, caps):
            binding.set_device_memory_cap(used + int(room))
            try:
                w2, k = launches(lambda: ctx.truncate(site, direction, D // 2, x))
            except binding.DMRGError as e:
                assert e.code == binding.ENOMEM
                assert binding.device_memory_in_use() == used
                refused.append(room)
                continue
            served.append(room)
            count.append(k)
            assert abs(w2 - w) <= 1e-12
            binding.set_device_memory_cap(0)
            assert np.abs(ctx.tt_to_x(site) - y).max() <= 1e-10
    finally:
        binding.set_device_memory_cap(0)
    assert refused and served and max(refused) < min(served)
    assert count[0] != refined and count[-1] == refined  # in place first, refined with room
