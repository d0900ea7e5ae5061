"""The autotuner times the SpMM kernels that a handle's routes launch: between
the spatial derivatives on the eigenbasis route, on three odd values on
Algorithm 1's, and the mixed modes' inner ones.  Whatever block sizes it picks,
every output is summed in the same order as with the fixed ones.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')


@pytest.mark.parametrize('m, prec, mk_route, names', [
    (13, 0, 0, ('apply_A grad', 'apply_even grad')),
    (14, 0, 1, ('apply_A', 'apply_even')),
    (15, 1, 0, ('apply_A grad', 'apply_even grad', 'apply_A fp32', 'apply_even fp32')),
    (17, 2, 0, ('apply_A grad', 'apply_even grad', 'apply_A bf16', 'apply_even fp32')),
    (18, 2, 1, ('apply_A', 'apply_even', 'apply_A bf16', 'apply_even fp32'))])
def test_tuned_kernels_are_those_that_run(m, prec, mk_route, names):
    import paper_2102_09038_gb300 as rte
    p = workloads.checkerboard(m=m, levels=2, g=0.8, ratio=0.9, blocks=1, nrhs=1)
    kw = dict(n_plus=2, n_minus=3, precision=prec, mk_route=mk_route)
    tuned, fixed = rte.Solver(p, autotune=1, **kw), rte.Solver(p, autotune=0, **kw)
    try:
        keys = [k for k in rte.autotune_report() if k.startswith('apply_') and ' m=%d ' % m in k]
        assert sorted(keys) == sorted('%s m=%d nS=64 rhs=1' % (n, m) for n in names)
        x = torch.tensor(np.random.default_rng(m).standard_normal((1, tuned.n_nodes, 64))).cuda()
        assert torch.equal(tuned.apply(x), fixed.apply(x))
        assert torch.equal(tuned.odd(x), fixed.odd(x))
    finally:
        tuned.close()
        fixed.close()
