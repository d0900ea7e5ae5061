"""The outer iteration's fused vector passes on vectors aligned for two values
at once and not: one cell, a partly filled block, several blocks a right-hand
side, one to three right-hand sides, no coarse space and one too wide for the
row kernels.

The two alignments add the dot products in another order, so their step
lengths agree to FP64 rounding; where that turns the rounding of an FP32 copy
the result moves by at most 2^-24 of an entry: 1e-7 of the largest.  The
solves are judged by the residual of the exact operator at twice the requested
tolerance, as a residual taken with another summation order.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')


def shifted(x, by):
    """x on the GPU, its first value `by` values past an allocation's start."""
    flat = torch.zeros(x.size + by, dtype=torch.float64, device='cuda')
    view = flat[by:].view(x.shape)
    view.copy_(torch.tensor(x))
    return view


@pytest.mark.parametrize('precision', [0, 1, 2])
@pytest.mark.parametrize('m, levels, nrhs, n_plus', [(1, 1, 1, 2), (3, 1, 3, 0), (8, 2, 2, 6),
                                                     (35, 2, 3, 4)])
def test_unaligned_vectors(m, levels, nrhs, n_plus, precision):
    import paper_2102_09038_gb300 as rte
    p = workloads.constant(m, levels, 0.6, 1.5, 1.2)
    s = rte.Solver(p, n_plus=n_plus, n_minus=3, precision=precision, max_rhs=nrhs,
                   e0_route=rte.E0_DIRECT)
    try:
        x = np.random.default_rng(m).standard_normal((nrhs, (m + 1) ** 2, 4 << (2 * levels)))
        for p2 in (False, True):
            got = []
            for by_in, by_out in ((0, 0), (1, 0), (0, 1)):
                out = shifted(np.zeros_like(x), by_out)
                s.precond(shifted(x, by_in), p2, out)
                got.append(out.cpu().numpy())
            for g in got[1:]:
                assert np.abs(g - got[0]).max() <= 1e-7 * np.abs(got[0]).max()
        for by in (0, 1):
            q, u = shifted(x, by), shifted(np.zeros_like(x), 1 - by)
            _, info = s.solve(q, u, tol=1e-9)
            assert info['status'] == 0
            res = (s.apply(u) - q).flatten(1).norm(dim=1) / q.flatten(1).norm(dim=1)
            assert res.max().item() <= 2e-9
    finally:
        s.close()


@pytest.mark.parametrize('precision', [1, 2])
def test_unaligned_vectors_on_the_multigrid_route(precision):
    # that route reads its right-hand side 16 bytes at a time; E_0 CG to 1e-5,
    # so the two results agree to a few times that
    import paper_2102_09038_gb300 as rte
    m, levels, nrhs = 9, 2, 2
    p = workloads.constant(m, levels, 0.6, 1.5, 1.2)
    s = rte.Solver(p, n_plus=2, n_minus=3, precision=precision, max_rhs=nrhs,
                   e0_route=rte.E0_MULTIGRID, e0_tol=1e-5)
    try:
        x = np.random.default_rng(m).standard_normal((nrhs, (m + 1) ** 2, 4 << (2 * levels)))
        got = []
        for by_in, by_out in ((0, 0), (1, 0), (0, 1), (1, 1)):
            out = shifted(np.zeros_like(x), by_out)
            s.precond(shifted(x, by_in), False, out)
            got.append(out.cpu().numpy())
        for g in got[1:]:
            assert np.abs(g - got[0]).max() <= 1e-4 * np.abs(got[0]).max()
    finally:
        s.close()


def test_p1_in_place():
    # the P_1 steps alone may write their result over their argument
    import paper_2102_09038_gb300 as rte
    p = workloads.constant(9, 2, 0.6, 1.5, 1.2)
    s = rte.Solver(p, n_plus=2, n_minus=3, precision=rte.MIXED_BF16, max_rhs=2)
    try:
        x = np.random.default_rng(5).standard_normal((2, 100, 64))
        want = s.precond(shifted(x, 0), False)
        got = shifted(x, 0)
        s.precond(got, False, got)
        assert (got - want).abs().max().item() <= 1e-7 * want.abs().max().item()
    finally:
        s.close()


@pytest.mark.parametrize('precision', [1, 2])
def test_unaligned_vectors_on_the_multigrid_route_of_p1_l(precision):
    # P_1^l hands the caller's vectors to E_0^{-1} themselves, as the operator
    # alone does; E_0 CG to 1e-5, the bound of the test above
    import paper_2102_09038_gb300 as rte
    m, levels, nrhs = 9, 2, 2
    p = workloads.constant(m, levels, 0.6, 1.5, 1.2)
    s = rte.Solver(p, n_plus=2, n_minus=3, precision=precision, max_rhs=nrhs, l=2,
                   p1_route=rte.P1_RICHARDSON, e0_route=rte.E0_MULTIGRID, e0_tol=1e-5)
    try:
        x = np.random.default_rng(m).standard_normal((nrhs, (m + 1) ** 2, 4 << (2 * levels)))
        for call in (lambda a, o: s.precond(a, False, o), lambda a, o: s.operator('E0_INV', a, o)):
            got = []
            for by_in, by_out in ((0, 0), (1, 0), (0, 1), (1, 1)):
                out = shifted(np.zeros_like(x), by_out)
                call(shifted(x, by_in), out)
                got.append(out.cpu().numpy())
            for g in got[1:]:
                assert np.abs(g - got[0]).max() <= 1e-4 * np.abs(got[0]).max()
    finally:
        s.close()
