"""The fp32 GEMM (tensor cores on exact bf16 triples) against an fp64 matmul: both orientations, K splits, edges of the
128-row / 32..128-column tiles and of the 32-wide K blocks, every epilogue."""
import pytest
import torch

pytestmark = pytest.mark.gpu

CASES = [
    # M, N, K
    (65, 32, 32, ), (128, 128, 128), (129, 97, 36), (384, 768, 768), (300, 2304, 100), (400, 96, 3072), (1000, 3072, 768),
    # swapped orientation: M <= 64
    (1, 128, 64), (16, 769, 3072), (32, 512, 256), (33, 1600, 1600), (64, 777, 260), (16, 50257, 768),
]


@pytest.mark.parametrize("M,N,K", CASES)
def test_f32_gemm_matches_fp64(M, N, K):
    import paper_2408_05636_b200 as sdd
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.rand(M + 5, K, device="cuda", generator=g) - 0.3      # a mean far from zero shows a biased accumulation
    W = torch.rand(N, K, device="cuda", generator=g) - 0.3
    bias = torch.randn(N, device="cuda", generator=g)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    plain = A[:M].double() @ W.double().t()
    for epi in (0, 1, 2, 3):
        for b in (bias, None):
            for ldc in (N + 3, (N + 7) // 4 * 4):                    # rows that are and are not 16-byte aligned
                out = torch.randn(M, ldc, device="cuda", generator=g)
                out0 = out.double().clone()
                torch.cuda.synchronize()
                sdd.sdd_debug_gemm_f32(A, W, b, M, epi, out, status)
                torch.cuda.synchronize()
                assert int(status.item()) == 0
                ref = plain if b is None else plain + b.double()
                if epi == 1:
                    ref = torch.nn.functional.gelu(ref, approximate="tanh")
                elif epi == 2:
                    ref = out0[:, :N] + ref
                err = (out[:, :N].double() - ref).norm() / ref.norm()
                assert err < 5e-7, (epi, ldc, float(err))
                assert torch.equal(out[:, N:].double(), out0[:, N:])     # nothing written past column N
