"""GPU: dmrg_truncate's eigensolver (FP32 Jacobi passes refined in FP64) against numpy's SVD
of the same two-site vector on small and large middle sectors, fast-falling, flat, degenerate
and rank-deficient spectra, both directions: the truncated state's projection onto x, the
discarded weight, and the normalisation of the factor the direction makes an isometry (the
energy of the truncated state through the operators, which assume it).

Tolerances.  Discarded weight and overlap: the Gram route has eigenvalue errors of ~1e-15 of
the largest, 1e-12 is asked.  A second truncation of the truncated vector to the same D
discards nothing (1e-12) and returns it (1e-10)."""
import numpy as np
import pytest

from tests.test_gpu_parity import Context  # noqa: F401  (fixture)
from workloads import hubbard_chain

pytestmark = pytest.mark.gpu


def vector(ctx, site, kind, seed):
    n, table = ctx.layout(site)
    rng = np.random.default_rng(seed)
    x = np.zeros(n)
    for row in table:
        dl, dr, off = int(row[9]), int(row[10]), int(row[11])
        if kind == "falling":
            b = rng.normal(size=(dl, dr)) * np.exp(-7.0 * np.arange(dl) / dl)[:, None] * np.exp(-5.0 * np.arange(dr) / dr)
        elif kind == "flat":
            b = rng.normal(size=(dl, dr))
        elif kind == "degenerate":
            b = np.eye(dl, dr)
        else:  # rank one
            b = np.outer(rng.normal(size=dl), rng.normal(size=dr))
        x[off:off + dl * dr] = b.ravel()
    return x / np.linalg.norm(x)


@pytest.mark.parametrize("L,D0", [(4, 3), (8, 40), (12, 500), (14, 1400)])
@pytest.mark.parametrize("kind", ["falling", "flat", "degenerate", "rank one"])
@pytest.mark.parametrize("direction", [1, -1])
def test_truncation_by_refined_eigenvectors(Context, L, D0, kind, direction):  # noqa: F811
    site = L // 2 - 1
    ctx = Context(L, [0] * L, L, 0, 0)
    ctx.set_integrals(*hubbard_chain(L, 1.0, 4.0))
    ctx.set_schedule([D0], [1e-8], [1], [0.0])
    ctx.init_mps(3)
    ctx.canonicalize(site)
    x = vector(ctx, site, kind, 5)
    # nothing to discard: the vector comes back
    assert abs(ctx.truncate(site, direction, 10 ** 9, x)) <= 1e-12
    y = ctx.tt_to_x(site)
    assert np.abs(y - x).max() <= 1e-10
    assert abs(np.linalg.norm(y) - 1.0) <= 1e-12
    # a cut: the kept part is the projection of x, its weight 1 - w_disc
    D = max(1, D0 // 3)
    w = ctx.truncate(site, direction, D, x)
    z = ctx.tt_to_x(site)
    assert abs(z @ x - (1.0 - w)) <= 1e-12
    assert abs(z @ z - (1.0 - w)) <= 1e-12
    e = ctx.energy(site, z)
    w2 = ctx.truncate(site, direction, D, z)
    assert abs(w2) <= 1e-12
    u = ctx.tt_to_x(site)
    assert np.abs(u * np.linalg.norm(z) - z).max() <= 1e-10
    # the isometry: operators of the grown block give the same energy at the next pair
    nxt = site + direction
    if 0 <= nxt <= L - 2:
        v = ctx.tt_to_x(nxt)
        assert abs(ctx.energy(nxt, v) - e) <= 1e-10 * max(1.0, abs(e))


def test_truncation_without_room_for_the_refined_solver(Context):  # noqa: F811
    """Under a device-memory cap that leaves room for the decomposition's own matrices only,
    the eigenproblems are solved in place and the result is the same state (1e-10)."""
    from paper_1312_2415_gb300 import binding
    L, D = 12, 400
    site = L // 2 - 1
    ctx = Context(L, [0] * L, L, 0, 0)
    ctx.set_integrals(*hubbard_chain(L, 1.0, 4.0))
    ctx.set_schedule([D], [1e-8], [1], [0.0])
    ctx.init_mps(3)
    ctx.canonicalize(site)
    x = vector(ctx, site, "falling", 5)
    w = ctx.truncate(site, 1, D // 2, x)
    y = ctx.tt_to_x(site)
    used = binding.device_memory_in_use()
    n = ctx.layout(site)[0]
    try:
        for room in (1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 64):  # multiples of the vector's bytes
            binding.set_device_memory_cap(used + room * 8 * n)
            try:
                w2 = ctx.truncate(site, 1, D // 2, x)
            except binding.DMRGError as e:
                assert e.code == binding.ENOMEM
                continue
            assert abs(w2 - w) <= 1e-12
            binding.set_device_memory_cap(0)
            assert np.abs(ctx.tt_to_x(site) - y).max() <= 1e-10
    finally:
        binding.set_device_memory_cap(0)
