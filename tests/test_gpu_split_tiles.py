"""The split FP64 GEMM over its tile widths, slice counts and ragged edges.

Exact: integers whose balanced base-128 digits fill the first D of S slices
with 2 D - 1 <= S lose no digit pair, so the product is the integer product
bit for bit while every slice pair (s, t) with s, t < D takes part (D = 2 for
S = 3, 4 and D = 3 for S >= 5; |x| <= 2^(7 D - 2) keeps all sums below 2^48,
which the double-float accumulation holds exactly).  A wrong pair, group,
tile edge, K tail or drain shows as a mismatch.
Accurate: random rows against FP64, within the dropped pairs' bound S K 2^-7S
of the row and column scales plus 2^-44.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')

# one row and column, K of one 16-byte piece; tiles one past an edge in each
# direction; K across the 512-term chunks; odd N (unaligned rows of C)
SHAPES = [(1, 1, 8), (129, 97, 24), (128, 96, 512), (257, 161, 520), (300, 33, 1048),
          (2500, 250, 72), (640, 385, 1544)]


def integers(rows, K, digits, seed):
    g = torch.Generator().manual_seed(seed)
    top = 1 << (7 * digits - 2)
    return torch.randint(-top, top + 1, (rows, K), generator=g).double()


@pytest.mark.parametrize('shape', SHAPES)
@pytest.mark.parametrize('slices', [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_exact_on_integers_of_several_digits(shape, slices):
    import paper_2102_09038_gb300 as rte
    M, N, K = shape
    D = 1 if slices < 3 else 2 if slices < 5 else 3
    A, B = integers(M, K, D, 7 * M + slices), integers(N, K, D, 5 * N + K)
    C = rte.dgemm_split(A.cuda(), B.cuda(), slices=slices).cpu()
    assert torch.equal(C, A @ B.T)


@pytest.mark.parametrize('shape', SHAPES)
@pytest.mark.parametrize('slices', [5, 6, 7, 9])
def test_random_rows_within_the_truncation_bound(shape, slices):
    import paper_2102_09038_gb300 as rte
    M, N, K = shape
    g = torch.Generator().manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g, dtype=torch.float64)
    A *= torch.logspace(-6, 6, M, dtype=torch.float64)[:, None]
    B = torch.randn(N, K, generator=g, dtype=torch.float64)
    C = rte.dgemm_split(A.cuda(), B.cuda(), slices=slices).cpu()
    scale = 4 * A.abs().amax(1)[:, None] * B.abs().amax(1)[None, :]   # 2^ea 2^eb
    err = ((C - A @ B.T).abs() / scale).max()
    assert err <= K * (slices * 2.0 ** (-7 * slices) + 2.0 ** -44), float(err)


def test_unaligned_operands_and_result():
    # contiguous tensors that start 8 bytes past an aligned address
    import paper_2102_09038_gb300 as rte
    M, N, K = 200, 96, 136
    g = torch.Generator().manual_seed(1)
    A = torch.randn(M * K + 1, generator=g, dtype=torch.float64).cuda()[1:].view(M, K)
    B = torch.randn(N * K + 1, generator=g, dtype=torch.float64).cuda()[1:].view(N, K)
    out = torch.zeros(M * N + 1, dtype=torch.float64, device='cuda')[1:].view(M, N)
    rte.dgemm_split_static(A, B, slices=7, out=out)
    ref = rte.dgemm_split(A.clone(), B.clone(), slices=7)
    assert torch.equal(out, ref)
