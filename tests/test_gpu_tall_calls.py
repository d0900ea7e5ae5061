"""FP64 contractions of calls with more row tiles than a grid's y dimension
holds: 2^21 rows (256 x 256 squares, 16 right-hand sides) by 32, 48 and 10
columns.  Every output sums over k in the same order whatever the call's tiles
and rows, so each right-hand side equals the call with it alone to the bit.
"""
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')


def test_right_hand_sides_of_a_tall_call():
    import paper_2102_09038_gb300 as rte
    m, nrhs = 256, 16
    s = rte.Solver(workloads.constant(m, 1, 0.6, 1.5, 1.2), n_plus=-1, n_minus=3, max_rhs=nrhs,
                   autotune=0)
    try:
        g = torch.Generator().manual_seed(3)
        x = torch.randn(nrhs, s.n_nodes, s.n_dirs, generator=g, dtype=torch.float64).cuda()
        z = torch.randn(1, s.n_cells, s.n_odd, generator=g, dtype=torch.float64).cuda().repeat(nrhs, 1, 1)
        y, u = s.apply(x), s.odd(x)
        prec = s.operator('MK_PREC', z, s.odd_zeros(nrhs))
        one = s.operator('MK_PREC', z[:1].clone(), s.odd_zeros(1))
        for r in (0, 7, nrhs - 1):
            xr = x[r:r + 1].clone()
            assert torch.equal(s.apply(xr)[0], y[r])
            assert torch.equal(s.odd(xr)[0], u[r])
            assert torch.equal(prec[r], one[0])
    finally:
        s.close()
