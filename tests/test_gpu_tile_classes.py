"""GPU: the tile classes of the mixed-precision matvec (tiny tiles on CUDA cores, tiles up to
32 x 32, up to 64 x 64 and larger on tensor cores, runs of terms summed in partial sums),
on states whose blocks straddle the classes' limits, against the same context's FP64 product.

Tolerance 2e-6 of the largest element: split TF32 keeps 22 significand bits per operand
(2.4e-7 per product) and sums of FP32 terms add a few times that."""
import numpy as np
import pytest

from tests.test_gpu_parity import Context  # noqa: F401  (fixture)
from workloads import hubbard_chain, random_integrals, round_robin_irreps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,L,N,tS,D,site", [
    ("random", 8, 8, 0, 40, 3), ("hubbard", 6, 6, 0, 5, 2), ("hubbard", 10, 10, 0, 150, 4),
    ("hubbard", 10, 10, 2, 420, 4), ("hubbard", 12, 12, 0, 900, 5), ("hubbard", 12, 12, 0, 1500, 5),
    ("hubbard", 14, 14, 0, 2600, 6), ("random", 12, 11, 1, 300, 4)])
def test_mixed_matvec_over_tile_classes(Context, kind, L, N, tS, D, site):  # noqa: F811
    irr = [0] * L if kind == "hubbard" else round_robin_irreps(L)
    ctx = Context(L, irr, N, tS, 0)
    ctx.set_integrals(*(hubbard_chain(L, 1.0, 4.0) if kind == "hubbard" else random_integrals(irr, 11)))
    ctx.set_schedule([D], [1e-8], [1], [0.0])
    ctx.init_mps(7)
    ctx.canonicalize(site)
    n, _ = ctx.layout(site)
    x = np.random.default_rng(D).normal(size=n)
    y = ctx.matvec(site, x)
    ctx.set_precision(1)
    z = ctx.matvec(site, x)
    assert np.array_equal(z, ctx.matvec(site, x))
    assert np.abs(z - y).max() <= 2e-6 * np.abs(y).max()
