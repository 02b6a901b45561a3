"""Hi/lo output pairs of the bf16 GEMM (GELU of the target's MLP) leaving by TMA: every tile width and the CTA-pair kernel,
ragged rows and columns, one and several tiles per CTA."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tile", [0, 64, 128, 256, 512])
@pytest.mark.parametrize("M,N,K", [(130, 200, 64), (999, 6400, 320), (3996, 1608, 192)])
def test_hi_lo_outputs(M, N, K, n_tile):
    import paper_2408_05636_b200 as sdd
    g = torch.Generator(device="cuda").manual_seed(M + n_tile)
    x = torch.randn(M + 9, K, device="cuda", generator=g)
    hi = x.to(torch.bfloat16)
    lo = (x - hi.float()).to(torch.bfloat16)
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.05).to(torch.bfloat16)
    bias = torch.randn(N, device="cuda", generator=g)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref = (hi[:M].float() + lo[:M].float()) @ W.float().t() + bias
    for epi, want in ((0, ref), (1, torch.nn.functional.gelu(ref, approximate="tanh"))):
        out = [torch.full((M, N + 8), 7.0, device="cuda", dtype=torch.bfloat16) for _ in range(2)]
        torch.cuda.synchronize()
        sdd.sdd_debug_gemm_bf16(hi, W, bias, M, epi, out[0], n_tile, True, status, None, lo, out[1])
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got = out[0][:, :N].float() + out[1][:, :N].float()
        assert (got - want).abs().max().item() < 2e-3 * max(1.0, want.abs().max().item())     # hardware tanh ~ 2^-11
        assert (out[0][:, N:] == 7).all() and (out[1][:, N:] == 7).all()                      # nothing past column N
