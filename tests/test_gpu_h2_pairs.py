"""The BF16 H^2 apply by pairs of outputs (k_h2_tc<2>): calls with rows enough
for the pairs against the same rows in calls short enough for single outputs.
Every output's products are summed in its list's order either way, so the
results are the same to the bit.  tests/test_host_h2_groups.py checks, with the
library's own rules, that these calls take the pairs and the short ones do not.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')

# levels, parity, groups of the smallest list taken by pairs, those lists
CALLS = [(3, -1, 6, ('near',)), (4, 1, 6, ('near', 'couple')), (4, -1, 6, ('near', 'couple')),
         (5, -1, 96, ('near',))]


def rows_for(groups, sms):
    """Rows from which every such list has two blocks per SM twice over, the
    last row tile partly filled."""
    return 128 * -(-4 * sms // groups) - 37


@pytest.mark.parametrize('levels, parity, groups, paired', CALLS)
def test_pairs_equal_single_outputs(levels, parity, groups, paired):
    import paper_2102_09038_gb300 as rte
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = rows_for(groups, sms)
    h = rte.H2Scattering(levels, 0.5, parities=1 if parity > 0 else 2, precisions=4)
    try:
        n = h.n_plus * (1 if parity > 0 else 3)
        g = torch.Generator().manual_seed(rows)
        X = torch.randn(rows, n, generator=g, dtype=torch.float64).cuda()
        Y = h.apply(X, parity=parity, precision=rte.MIXED_BF16)
        for a, b in ((0, 128), (128, 129), (rows // 2, rows // 2 + 100), (rows - 91, rows)):
            Z = h.apply(X[a:b], parity=parity, precision=rte.MIXED_BF16)
            assert torch.equal(Z, Y[a:b])
    finally:
        h.close()
