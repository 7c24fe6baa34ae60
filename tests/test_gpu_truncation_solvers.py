"""Eqs. 26-28 by the FP64 Jacobi solver of sweep steps (dmrg_truncate has a solver of its own)
and by dmrg_truncate on nearly degenerate spectra, against the oracle's numpy SVD of the same
blocks: the discarded weight (Eq. 15) and the truncated two-site tensor, which does not depend
on the bases the solvers choose inside a degenerate cluster.

A sweep step whose Davidson stops at its first iteration decomposes the state it was given: one
with chosen singular values between the singular vectors of a random two-site tensor.  In every
sector half of the values lie above a gap, at which the state is cut: evenly spread ones, and
two clusters at 1 and 1/2 of squared values delta apart.  Tolerance: the Davis-Kahan bound of
the Gram route (truncation_bound), which is 1e-12 here."""
import numpy as np
import pytest

from oracle import mps as om
from tests.mps_io import lib_x_to_oracle, mps_to_bytes, oracle_x_to_lib, truncation_bound
from tests.test_gpu_parity import Context  # noqa: F401  (fixture)
from workloads import hubbard_chain, uniform_pm1

pytestmark = pytest.mark.gpu
L = N = 12
SITE = L // 2 - 1


@pytest.fixture(scope="module", params=[300, 1500], ids=["up to 64 rows", "up to 210 rows"])
def state(request):
    D = request.param
    m = om.right_canonicalize(om.random_mps([0] * L, N, 0, 0, D, uniform_pm1(12, 10 ** 7)))
    for k in range(SITE):
        om.svd_truncate(m, k, om.tt_to_x(m, k), 10 ** 9, "right")
    return D, m


def chosen(m, table, n, kind):
    """m with the middle bond of sites SITE, SITE + 1 replaced: (state, kept above the gap)."""
    g = lib_x_to_oracle(np.random.default_rng(5).normal(size=n), table)
    left, right = m.copy(), m.copy()
    om.svd_truncate(left, SITE, g, 10 ** 9, "right")  # T[SITE] = U
    om.svd_truncate(right, SITE, g, 10 ** 9, "left")  # T[SITE + 1] = V
    kept, values = 0, {}
    for sec, r in left.dims[SITE + 1].items():
        h, k = (r + 1) // 2, np.arange(r)
        kept += h
        if kind == "spread":
            values[sec] = np.where(k < h, 1.0 - 0.4 * k / h, 0.4 - 0.3 * (k - h) / r)
        else:
            values[sec] = np.sqrt(np.where(k < h, 1.0, 0.25) * (1.0 - kind * k))
    left.T[SITE + 1] = {k: values[k[1]][:, None] * b for k, b in right.T[SITE + 1].items()}
    return left, kept


def setup(Context, state, kind):  # noqa: F811
    D, m = state
    ctx = Context(L, [0] * L, N, 0, 0)
    ctx.set_integrals(*hubbard_chain(L, 1.0, 4.0))
    ctx.set_schedule([D], [0.0], [1], [0.0], 1e-14, 1)
    ctx.set_mps(mps_to_bytes(m))
    n, table = ctx.layout(SITE)
    made, kept = chosen(m, table, n, kind)
    x = oracle_x_to_lib(om.tt_to_x(made, SITE), table, n)
    return ctx, made, table, n, x / np.linalg.norm(x), kept


def compare(ctx, m, table, n, x, D, direction, w):
    """The state in ctx against the SVD truncation of x to D values; w: its discarded weight."""
    m2 = m.copy()
    w_o, _, groups = om.svd_truncate(m2, SITE, lib_x_to_oracle(x, table), D, "right" if direction > 0 else "left")
    tol = truncation_bound(groups, D)
    assert tol < 2e-12, (D, tol)
    assert abs(w - w_o) < 1e-12, (D, w, w_o)
    got, want = ctx.tt_to_x(SITE), oracle_x_to_lib(om.tt_to_x(m2, SITE), table, n)
    assert np.abs(got - want).max() < tol, (D, np.abs(got - want).max(), tol)


@pytest.mark.parametrize("kind", ["spread", 1e-6])
@pytest.mark.parametrize("direction", [1, -1])
def test_sweep_step_against_svd(Context, state, kind, direction):  # noqa: F811
    ctx, m, table, n, x, kept = setup(Context, state, kind)
    for Dt in (kept, 10 ** 6):
        ctx.set_mps(mps_to_bytes(m))
        assert np.abs(ctx.tt_to_x(SITE) / np.linalg.norm(ctx.tt_to_x(SITE)) - x).max() < 1e-13
        _, w, _, _ = ctx.sweep_step(SITE, direction, Dt)
        compare(ctx, m, table, n, x, Dt, direction, w)


@pytest.mark.parametrize("kind", ["spread", 3e-8, 1e-6, 5e-6, 3e-5])
@pytest.mark.parametrize("direction", [1, -1])
def test_truncate_against_svd(Context, state, kind, direction):  # noqa: F811
    ctx, m, table, n, x, kept = setup(Context, state, kind)
    for Dt in (kept, 10 ** 6):
        w = ctx.truncate(SITE, direction, Dt, x)
        compare(ctx, m, table, n, x, Dt, direction, w)
