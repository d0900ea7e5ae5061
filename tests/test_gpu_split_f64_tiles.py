"""The FP64 GEMM's tile choice and the digit split's row blocks: products that
do not depend on how many rows the call has.

FP64 GEMM: E u of one right-hand side against the same one among three, which
takes other tiles: every output sums over k in one order, so bit by bit; the
meshes and spheres reach each of the four tiles, whole and ragged.  Digit
split: integers of two digits at four slices lose no digit pair (their sums
stay below 2^48), so the product is the integer product; rows below, at and
past a block, both sides of each line of the block rule, K of one 16-byte
piece up to many.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')


@pytest.mark.parametrize('m, levels', [(1, 0), (5, 1), (9, 3), (17, 2), (24, 3), (33, 2), (48, 1)])
def test_fp64_operator_does_not_depend_on_the_tile(m, levels):
    import paper_2102_09038_gb300 as rte
    p = workloads.constant(m, levels, 0.6, 1.5, 1.2)
    s = rte.Solver(p, n_plus=0, n_minus=1, max_rhs=3, dgemm=rte.DGEMM_SIMT)
    try:
        x = torch.tensor(np.random.default_rng(m).standard_normal(
            (3, (m + 1) ** 2, 4 << (2 * levels))), device='cuda')
        all3 = s.apply(x)
        for r in range(3):
            assert torch.equal(s.apply(x[r:r + 1].contiguous()), all3[r:r + 1])
    finally:
        s.close()


@pytest.mark.parametrize('K', [8, 504, 520, 3072])
@pytest.mark.parametrize('M', [1, 7, 9, 2431, 2440, 9727, 9760])
def test_split_rows_and_threads(M, K):
    import paper_2102_09038_gb300 as rte
    g = torch.Generator().manual_seed(M + K)
    A = torch.randint(-4096, 4097, (M, K), generator=g).double().cuda()
    B = torch.randint(-4096, 4097, (40, K), generator=g).double().cuda()
    assert torch.equal(rte.dgemm_split(A, B, slices=4), A @ B.T)
