"""rte_destroy waits for the handle's own stream and for nothing else: a handle
closed while another stream is busy for half a second is gone before that
stream is done (the server evicts idle handles while its other slots solve)."""
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')


@pytest.mark.parametrize('prec', [0, 2])
def test_destroy_does_not_wait_for_other_streams(prec):
    import paper_2102_09038_gb300 as rte
    p = workloads.constant(8, 1, 0.7, 1.0, 0.9)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    q = torch.tensor(p.q_nodal, dtype=torch.float64, device='cuda')
    A = torch.randn(8192, 8192, device='cuda')
    A @ A
    torch.cuda.synchronize()
    for _ in range(2):   # the first handle of a process loads the kernels
        s = rte.Solver(p, stream=mine, n_plus=2, n_minus=3, precision=prec, autotune=0)
        u, info = s.solve(s.rhs(q), tol=1e-8)
        assert info['status'] == 0
        mine.synchronize()
        done = torch.cuda.Event()
        with torch.cuda.stream(other):
            for _ in range(40):
                A @ A
            done.record()
        s.close()
        busy = not done.query()
        torch.cuda.synchronize()
    assert busy
