"""GPU: the grouped FP64 block products at the edges of their work split (blocks of one row
up to several 32-lane slices, one task up to lists shared by eight warps), through the
matvec, the allocation-free matvec and the energy, against the oracle's dense H_eff.

Tolerance 1e-12 of the largest element: sums of up to ~1e4 rounded products of O(1) terms
in FP64 are off by ~1e-14 whatever the order of summation."""
import numpy as np
import pytest

from oracle import dmrg as odmrg
from tests.mps_io import lib_x_to_oracle, mps_to_bytes, oracle_x_to_lib
from tests.test_gpu_parity import Context, setup  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,L,N,tS,D,site", [
    ("hubbard", 4, 4, 0, 1, 1), ("random", 5, 5, 1, 3, 0), ("hubbard", 8, 8, 0, 17, 4), ("random", 7, 7, 1, 33, 5),
    ("hubbard", 8, 8, 2, 130, 3), ("hubbard", 8, 6, 0, 400, 3), ("random", 8, 8, 0, 90, 3)])
def test_matvec_and_energy_over_block_sizes(Context, kind, L, N, tS, D, site):  # noqa: F811
    import torch
    irr, h, V, m, prob = setup(kind, L, N, tS, 0, D, 5, site)
    H, _, proj = odmrg.effective_hamiltonian(prob, m, site)
    ctx = Context(L, irr, N, tS, 0)
    ctx.set_integrals(h, V)
    ctx.set_mps(mps_to_bytes(m))
    n, table = ctx.layout(site)
    v = np.random.default_rng(D).normal(size=n)
    yo = H @ proj.flatten(lib_x_to_oracle(v, table))
    want = oracle_x_to_lib(proj.unflatten(yo), table, n)
    tol = 1e-12 * np.abs(want).max()
    assert np.abs(ctx.matvec(site, v) - want).max() <= tol
    x = torch.tensor(v, device="cuda")
    y = torch.full_like(x, 7.0)
    torch.cuda.synchronize()
    ctx.matvec_noalloc(site, x.data_ptr(), y.data_ptr(), 0)
    torch.cuda.synchronize()
    assert np.abs(y.cpu().numpy() - want).max() <= tol
    assert abs(ctx.energy(site, x) - v @ want / (v @ v)) <= 1e-12 * np.linalg.norm(want) / np.linalg.norm(v)
