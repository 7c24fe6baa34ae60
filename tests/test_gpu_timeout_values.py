"""GPU: what a mixed-precision matvec whose waits time out (test hook) leaves in y.  The call fails
with DMRG_ECUDA; y is not the product, but it is made of numbers the library has written, not of
what device memory held before: the tables are built where a product with NaN was computed."""
import numpy as np
import pytest

from tests.test_gpu_parity import Context  # noqa: F401  (fixture)
from workloads import hubbard_chain

pytestmark = pytest.mark.gpu


def test_timed_out_matvec_leaves_numbers(Context):  # noqa: F811
    import torch
    from paper_1312_2415_gb300 import binding
    L, site = 12, 5
    ctx = Context(L, [0] * L, L, 0, 0, precision=1)
    ctx.set_integrals(*hubbard_chain(L, 1.0, 4.0))
    ctx.set_schedule([300], [0.0], [1], [0.0], 1e-10, 20)
    ctx.init_mps(1)
    ctx.canonicalize(site)
    mps = ctx.get_mps()
    n, _ = ctx.layout(site)
    x = torch.ones(n, dtype=torch.float64, device="cuda")
    y = torch.empty_like(x)
    ctx.matvec(site, x, y)
    assert torch.isfinite(y).all()
    ref = y.clone()
    ctx.matvec(site, torch.full_like(x, float("nan")), y)
    assert torch.isnan(y).any()
    ctx.set_mps(mps)  # frees the tables
    try:
        binding.test_tc_timeout(1)
        with pytest.raises(binding.DMRGError) as e:
            ctx.matvec(site, x, y)
        assert e.value.code == binding.ECUDA
        assert torch.isfinite(y).all()
        v = ctx.tt_to_x(site)
        with pytest.raises(binding.DMRGError) as e:
            ctx.davidson(site, v)
        assert e.value.code == binding.ECUDA and np.isfinite(v).all()
    finally:
        binding.test_tc_timeout(0)
    ctx.matvec(site, x, y)
    assert torch.equal(y, ref)
