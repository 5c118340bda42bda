"""Projections with few outputs and a long K around the row counts where the
cluster split-K kernel hands over to pairs of SMs: on either side a row has the
bits it has in a small launch, and the value of the 64-bit product."""
import pytest

pytestmark = pytest.mark.gpu


# (N, K): feed-forward out and history projection of the tiny and large widths,
# attention out, clusters of 16 with room for two token tiles
@pytest.mark.parametrize("N,K", [(384, 1536), (384, 1920), (1280, 6400), (1280, 5120), (1280, 1280), (768, 3072)])
def test_rows_are_the_same_on_both_sides_of_the_handover(N, K):
    import torch
    from paper_2609_32869_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(N + K)
    M = 257
    x = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    w = (0.02 * torch.randn(N, K, generator=g, device="cuda")).bfloat16()
    b = (0.02 * torch.randn(N, generator=g, device="cuda")).bfloat16()

    def run(lo, hi):
        y = torch.full((hi - lo, N), float("nan"), device="cuda")
        B.wf_gemm_bf16(x[lo:hi], w, b, y, hi - lo, N, K, None, 0)
        return y

    want = torch.cat([run(lo, min(M, lo + 40)) for lo in range(0, M, 40)])
    for m in (96, 97, 112, 113, 128, 129, 192, 193, 256, M):
        assert torch.equal(run(0, m), want[:m]), m
    bound = K * 2.0 ** -23 * (x.double().abs() @ w.double().abs().T) + 1e-6
    assert ((want.double() - (x.double() @ w.double().T + b.double())).abs() <= bound).all()
