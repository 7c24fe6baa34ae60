"""GPU: the vectors of a batched matvec are copied as one copy call per instance would, in
order: buffers of the batch passed as another instance's vector, an instance given twice, one
output for two instances, vectors at an odd address and vectors in pinned host memory.  Whole
results are compared bit for bit with runs on plain device vectors."""
import ctypes

import numpy as np
import pytest

from tests.test_gpu_batch import mods  # noqa: F401  (fixture)
from workloads import hubbard_chain

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctxs(mods):  # noqa: F811
    torch, Batch, Context, DMRGError = mods
    out = []
    for seed in (1, 2, 3):
        c = Context(12, [0] * 12, 12, 0, 0)
        c.set_integrals(*hubbard_chain(12, 1.0, 4.0))
        c.set_schedule([300], [0.0], [1], [0.0])
        c.init_mps(seed)
        c.canonicalize(5)
        out.append(c)
    return out


def run(lib, b, xs, ys):
    import torch
    n = len(xs)
    rc = lib.dmrg_batch_run(b.h, (ctypes.c_void_p * n)(*xs), (ctypes.c_void_p * n)(*ys), 1)
    assert rc == 0, lib.dmrg_batch_last_error(b.h)
    torch.cuda.synchronize()


def test_copies_keep_their_order(mods, ctxs):  # noqa: F811
    torch, Batch, Context, DMRGError = mods
    lib = ctxs[0].lib
    b = Batch(ctxs, [5, 5, 5], autotune=False)
    n = b.io(0)[2]
    assert all(b.io(i)[2] == n for i in range(3))
    g = torch.Generator(device="cuda").manual_seed(7)
    v = [torch.randn(n, dtype=torch.float64, device="cuda", generator=g) for _ in range(3)]
    y = [torch.empty_like(v[0]) for _ in range(3)]
    ptr = [t.data_ptr() for t in v]
    out = [t.data_ptr() for t in y]

    def want(order):
        run(lib, b, [ptr[k] for k in order], out)
        return [t.clone() for t in y]
    for _ in range(4):
        # the batch's own inputs as vectors: instance 0 takes 1's, then 1 takes 0's (by now
        # 1's), then 2 takes 0's
        ref = want((1, 1, 1))
        run(lib, b, ptr, out)
        bx = [b.io(i)[0] for i in range(3)]
        run(lib, b, [bx[1], bx[0], bx[0]], out)
        assert all(torch.equal(a, r) for a, r in zip(y, ref))
        # one output for all: the last instance's
        ref = want((0, 1, 2))
        run(lib, b, ptr, [out[0]] * 3)
        assert torch.equal(y[0], ref[2])
    # odd addresses and pinned host memory
    raw = torch.empty(8 * n + 8, dtype=torch.uint8, device="cuda")
    for off in (4, 1):
        raw[off:off + 8 * n] = v[1].view(torch.uint8)
        run(lib, b, [ptr[0], raw.data_ptr() + off, ptr[2]], out)
        assert all(torch.equal(a, r) for a, r in zip(y, ref))
        run(lib, b, ptr, [out[0], raw.data_ptr() + off, out[2]])
        assert torch.equal(raw[off:off + 8 * n].clone().view(torch.float64), ref[1])
    hx, hy = [t.cpu().pin_memory() for t in v], torch.zeros(n, dtype=torch.float64).pin_memory()
    run(lib, b, [t.data_ptr() for t in hx], [out[0], hy.data_ptr(), out[2]])
    assert torch.equal(hy, ref[1].cpu()) and torch.equal(y[0], ref[0]) and torch.equal(y[2], ref[2])
    b.close()


def test_an_instance_given_twice(mods, ctxs):  # noqa: F811
    torch, Batch, Context, DMRGError = mods
    lib = ctxs[0].lib
    b = Batch([ctxs[0], ctxs[0]], [5, 5], autotune=False)
    n = b.io(0)[2]
    v = [torch.tensor(np.random.default_rng(k).normal(size=n), device="cuda") for k in range(2)]
    y = [torch.empty_like(v[0]) for _ in range(2)]
    out = [t.data_ptr() for t in y]
    run(lib, b, [v[1].data_ptr()] * 2, out)
    ref = y[1].clone()
    for _ in range(4):
        run(lib, b, [v[0].data_ptr(), v[1].data_ptr()], out)
        assert torch.equal(y[0], ref) and torch.equal(y[1], ref)
    b.close()
