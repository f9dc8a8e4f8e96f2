"""The FMA contraction kernel in isolation (debug entry point of the C ABI) against fp64 numpy: both tile sizes, edges of
tiles and k slices, contractions shared by a cluster of blocks, rows that are not 16-byte aligned, every operand order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a_k,b_k", [(1, 1), (1, 0), (0, 0), (0, 1)])
@pytest.mark.parametrize("M,N,K,ld_extra", [(1, 1, 1, 0), (32, 32, 128, 0), (33, 40, 129, 0), (256, 40, 128, 4), (128, 32, 600, 0),
                                            (70, 36, 2048, 0), (63, 65, 1030, 3), (1500, 900, 40, 0), (1400, 1100, 700, 1)])
@pytest.mark.parametrize("accumulate", [0, 1])
def test_fp32_contraction(a_k, b_k, M, N, K, ld_extra, accumulate):
    import torch
    from paper_2502_16927_b200 import binding

    g = np.random.default_rng(M + 7 * N + K)
    a = g.standard_normal((M, K)).astype(np.float32)
    b = g.standard_normal((N, K)).astype(np.float32)
    c0 = g.standard_normal((M, N)).astype(np.float32)

    def place(x):
        rows, cols = x.shape
        t = torch.full((rows, cols + ld_extra), float("nan"), device="cuda")
        t[:, :cols] = torch.from_numpy(x).cuda()
        return t

    A, B, C = place(a if a_k else np.ascontiguousarray(a.T)), place(b if b_k else np.ascontiguousarray(b.T)), place(c0)
    layer = binding.Layer(64, 64, 64, 8, 1, 16, binding.BIGMAC_F32, 0)
    q = binding.bigmac_debug_gemm_t(A=A.data_ptr(), B=B.data_ptr(), C=C.data_ptr(), lda=A.shape[1], ldb=B.shape[1], ldc=C.shape[1],
                                    M=M, N=N, K=K, a_kmajor=a_k, b_kmajor=b_k, accumulate=accumulate)
    binding.bigmac_debug_gemm(layer.handle, q, 0)
    torch.cuda.synchronize()
    ref = a.astype(np.float64) @ b.astype(np.float64).T + (c0 if accumulate else 0)
    got = C.cpu().numpy()
    # K fp32 products of unit variance, summed: rounding of at most about K/2 steps of 2^-24 of the running sum
    assert np.max(np.abs(got[:, :N] - ref)) <= 2.0 ** -23 * (K ** 0.5 + 4) * (K ** 0.5) + 1e-6
    assert np.all(np.isnan(got[:, N:]))
    layer.close()
