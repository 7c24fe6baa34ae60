"""GPU: the mixed-precision matvec where its partial sums (one float per output element and 16
terms) do not fit under the device-memory cap beside its other tables: the output tiles go in
passes that share a smaller array, and y is the same to the bit, alone and in a batch.  With
room for half of the tables the call fails and leaves no device bytes behind."""
import pytest

from tests.test_gpu_parity import Context  # noqa: F401  (fixture)
from workloads import make_problem

pytestmark = pytest.mark.gpu


def test_partial_sums_in_passes(Context):  # noqa: F811
    import torch
    from paper_1312_2415_gb300 import Batch, binding
    cfg, h, V = make_problem("random28")
    D, site = 1500, cfg["L"] // 2 - 1
    ctx = Context(cfg["L"], cfg["group_irreps"], cfg["N"], cfg["two_S"], cfg["irrep"], group=7)
    ctx.set_integrals(h, V)
    ctx.set_schedule([D], [0.0], [1], [0.0])
    ctx.init_mps(1)
    ctx.canonicalize(site)
    mps = ctx.get_mps()
    n, _ = ctx.layout(site)
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    y = torch.empty_like(x)

    def fp64_plan():
        ctx.set_precision(0)
        ctx.set_mps(mps)  # drops the tables
        ctx.matvec(site, x, y)
        ctx.set_precision(1)
        return binding.device_memory_in_use()

    def launches(f):
        a = ctx.stats()["kernels_launched"]
        f()
        return ctx.stats()["kernels_launched"] - a
    before = fp64_plan()
    ctx.matvec(site, x, y)
    ref, tables = y.clone(), binding.device_memory_in_use() - before
    one_pass = launches(lambda: ctx.matvec(site, x, y))
    try:
        for share in (0.97, 0.96):
            assert fp64_plan() == before
            binding.set_device_memory_cap(before + int(share * tables))
            ctx.matvec(site, x, y)
            assert binding.device_memory_in_use() <= before + share * tables
            assert torch.equal(y, ref)
            y.fill_(7.0)
            assert launches(lambda: ctx.matvec(site, x, y)) > one_pass
            assert torch.equal(y, ref)
            binding.set_device_memory_cap(0)
        alone = binding.device_memory_in_use()
        Batch([ctx], [site], autotune=False).close()  # a first one: as the second, all else made
        b = Batch([ctx], [site], autotune=False)
        extra = binding.device_memory_in_use() - alone
        b.close()
        binding.set_device_memory_cap(alone + int(0.9 * extra))
        b = Batch([ctx], [site], autotune=False)
        binding.set_device_memory_cap(0)
        assert binding.device_memory_in_use() <= alone + 0.9 * extra
        y.fill_(7.0)
        b.run([x], [y])
        torch.cuda.synchronize()
        assert torch.equal(y, ref)
        b.close()
        assert fp64_plan() == before
        binding.set_device_memory_cap(before + tables // 2)
        with pytest.raises(binding.DMRGError) as e:
            ctx.matvec(site, x, y)
        assert e.value.code == binding.ENOMEM
        assert binding.device_memory_in_use() == before
    finally:
        binding.set_device_memory_cap(0)
