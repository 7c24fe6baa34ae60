"""GPU: the small Rayleigh-Ritz eigenproblems inside Davidson, through runs whose subspace grows
to every size up to a restart, on separated, nearly degenerate and exactly degenerate spectra,
against the oracle's dense eigenvalues.

Tolerances: residual 1e-10 gives an eigenvalue error below 1e-18 / gap plus rounding, 1e-10
is asked; the vector's own residual through the oracle's H_eff stays below 1e-9."""
import numpy as np
import pytest

from oracle import dmrg as odmrg
from tests.mps_io import lib_x_to_oracle, mps_to_bytes
from tests.test_gpu_parity import Context, setup  # noqa: F401  (fixture)
from workloads import hubbard_chain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N,tS,D,site,U", [(2, 2, 0, 4, 0, 4.0), (4, 4, 0, 3, 1, 4.0), (4, 4, 2, 20, 1, 0.0),
                                             (6, 6, 0, 60, 2, 0.0), (6, 6, 0, 60, 2, 1e-7), (6, 6, 0, 60, 2, 1e3),
                                             (8, 8, 0, 40, 3, 4.0)])
def test_davidson_eigenpairs(Context, L, N, tS, D, site, U):  # noqa: F811
    irr, _, _, m, _ = setup("hubbard", L, N, tS, 0, D, 9, site)
    h, V = hubbard_chain(L, 1.0, U)
    H, _, proj = odmrg.effective_hamiltonian(odmrg.Problem(h, V, irr, N, tS, 0), m, site)
    ctx = Context(L, irr, N, tS, 0)
    ctx.set_integrals(h, V)
    ctx.set_mps(mps_to_bytes(m))
    ctx.set_schedule([D], [1e-8], [1], [0.0], davidson_tol=1e-10 * max(1.0, U / 4.0), davidson_max_iter=400)
    n, table = ctx.layout(site)
    x = np.random.default_rng(3).normal(size=n)
    e, _, ok = ctx.davidson(site, x)
    scale = max(1.0, U / 4.0)
    w = np.linalg.eigvalsh(H)
    assert ok and abs(e - w[0]) <= 1e-10 * scale
    v = proj.flatten(lib_x_to_oracle(x, table))
    assert abs(v @ v - 1.0) <= 1e-12
    assert np.linalg.norm(H @ v - e * v) <= 1e-9 * scale
