"""The H^2 apply's row-tile and output-group choices: a call with many rows
(64 x 64 tiles; on the tensor cores four outputs a block) against calls with
its first 1, 33, 65 and 130 rows (smaller tiles; one output a block), which
the oracle tests cover.  Every choice sums the same products, so the bounds
are those tests': 1e-12, 2e-5 and 4 unit roundoffs of BF16 of the largest
entry.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')


@pytest.mark.parametrize('levels, parity, rows', [(3, 1, 19500), (3, -1, 6600), (4, 1, 4900),
                                                  (4, -1, 1700), (5, 1, 1300), (5, -1, 600)])
def test_rows_do_not_depend_on_the_call(levels, parity, rows):
    import paper_2102_09038_gb300 as rte
    h = rte.H2Scattering(levels, 0.5, parities=1 if parity > 0 else 2)
    try:
        n = h.n_plus * (1 if parity > 0 else 3)
        g = torch.Generator().manual_seed(rows)
        X = torch.randn(rows, n, generator=g, dtype=torch.float64).cuda()
        for prec, tol in ((rte.FP64, 1e-12), (rte.MIXED_FP32, 2e-5), (rte.MIXED_BF16, 4 * 2.0 ** -9)):
            Y = h.apply(X, parity=parity, precision=prec)
            for sub in (1, 33, 65, 130):
                Z = h.apply(X[:sub], parity=parity, precision=prec)
                assert (Z - Y[:sub]).abs().max().item() <= tol * Y.abs().max().item()
            # and the last rows, which end in a partly filled tile
            Z = h.apply(X[rows - 40:], parity=parity, precision=prec)
            assert (Z - Y[rows - 40:]).abs().max().item() <= tol * Y.abs().max().item()
    finally:
        h.close()
