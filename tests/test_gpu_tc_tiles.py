"""The tensor-core GEMM where a block walks several tiles: one to three tiles a
block, both accumulators reused, one stage of K up to several rounds of the
ring, remainders in M, N and K.

Entries j/64, |j| <= 64, are exact in BF16 and TF32 and the FP32 sums of their
products are exact, so the result is the FP64 product itself.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip('torch')


@pytest.mark.parametrize('bf16, out_bf16', [(True, False), (True, True), (False, False)])
@pytest.mark.parametrize('M, N, K', [(40000, 72, 8), (40000, 128, 64), (20011, 300, 72),
                                     (9000, 1030, 328), (58369, 130, 40)])
def test_many_tiles_a_block(M, N, K, bf16, out_bf16):
    import paper_2102_09038_gb300 as rte
    g = torch.Generator().manual_seed(M + N + K)
    A = torch.randint(-64, 65, (M, K), generator=g).double().cuda() / 64
    B = torch.randint(-64, 65, (N, K), generator=g).double().cuda() / 64
    ref = A @ B.T
    dt = torch.bfloat16 if bf16 else torch.float32
    C = rte.gemm_lowp(A.to(dt), B.to(dt), out_bf16=out_bf16)
    assert torch.equal(C, ref.to(C.dtype))
