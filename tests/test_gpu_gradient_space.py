"""E u and the odd part through the spatial derivatives (W = [A_1 A_2]^T V in
place of V on three odd values) at the edges: one cell, four directions, both
FP64 GEMM routes, vectors that are aligned for two values at once and not.

Against the oracle's operators at the parity tests' 1e-11 of direct applies
(max norm); the two alignments take the same steps and agree bit by bit.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')


def shifted(x, by):
    """x on the GPU, its first value `by` values past an allocation's start."""
    flat = torch.zeros(x.size + by, dtype=torch.float64, device='cuda')
    view = flat[by:].view(x.shape)
    view.copy_(torch.tensor(x))
    return view


@pytest.mark.parametrize('split', [False, True])
@pytest.mark.parametrize('m, levels, nrhs', [(1, 0, 1), (1, 1, 3), (2, 0, 2), (5, 1, 2), (12, 2, 1)])
def test_apply_and_odd_part(m, levels, nrhs, split):
    import paper_2102_09038_gb300 as rte
    p = workloads.constant(m, levels, 0.6, 1.5, 1.2)
    p.sigma_t[: m * m] *= 3.0
    disc = oracle.Discretisation(p.m, p.levels, p.sigma_t, p.sigma_s, p.g)
    ops = oracle.Operators(disc, n_plus=2, n_minus=3)
    s = rte.Solver(p, n_plus=0, n_minus=1, max_rhs=nrhs,
                   dgemm=rte.DGEMM_SPLIT if split else rte.DGEMM_SIMT, split_slices=9)
    try:
        x = np.random.default_rng(m).standard_normal((nrhs, disc.nRp, disc.nSp))
        if split and levels == 0:   # 12 odd columns, not a multiple of 8: refused
            with pytest.raises(rte.RteError):
                s.apply(shifted(x, 0))
            with pytest.raises(rte.RteError):
                s.odd(shifted(x, 0))
            return
        run_e = lambda v, out: s.operator('E', v, out)
        for run, ref in ((run_e, ops.apply_E), (s.apply, ops.apply_EK)):
            want = np.stack([ref(v) for v in x])
            got = []
            for by_in, by_out in ((0, 0), (1, 0), (0, 1), (1, 1)):
                out = shifted(np.zeros_like(x), by_out)
                run(shifted(x, by_in), out)
                got.append(out.cpu().numpy())
            assert np.abs(got[0] - want).max() < 1e-11 * np.abs(want).max()
            assert all(np.array_equal(g, got[0]) for g in got[1:])
        want = np.stack([ops.solve_MKminus(-ops.apply_A(v)) for v in x])
        u0, u1 = (s.odd(shifted(x, by)).cpu().numpy() for by in (0, 1))
        assert np.abs(u0 - want).max() < 1e-11 * np.abs(want).max()
        assert np.array_equal(u0, u1)
        zero = torch.zeros(want.shape, dtype=torch.float64, device='cuda')
        given = s.odd(shifted(x, 0), zero).cpu().numpy()
        assert np.abs(given - want).max() < 1e-11 * np.abs(want).max()
    finally:
        s.close()
