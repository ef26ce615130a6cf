"""The tensor-core GEMM on pairs of CTAs (more than 128 columns): column counts
that are and are not multiples of 32, odd numbers of 128-row halves, tiles whole
and split between pairs, a wider C; B rows behind the last are NaN and must not
enter.  Against the FP64 product of the same BF16 inputs; tolerance as in the
GEMM's other tests (FP32 accumulation of up to 8192 products of random signs,
1e-5 of the largest entry)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [144, 160, 176, 208, 224, 240])
@pytest.mark.parametrize("M,K,wide", [(128, 64, 0), (384, 512, 0), (38528, 64, 0), (384, 8192, 0), (1152, 4096, 12),
                                      (640, 1536, 3)])
def test_pairs(N, M, K, wide):
    from paper_2104_04609_gb300 import binding as B

    g = torch.Generator(device="cpu").manual_seed(M + K + N)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16).cuda()
    Bb = torch.full((256, K), float("nan"), dtype=torch.bfloat16, device="cuda")
    Bb[:N] = torch.randn(N, K, generator=g).to(torch.bfloat16).cuda()
    Bm = Bb[:N]
    Cw = torch.full((M, N + wide), float("nan"), dtype=torch.float32, device="cuda")
    C = Cw[:, :N]
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    nb = B.osrc_gemm_bf16_ws_bytes(M, N, K)
    ws = torch.full((max(nb, 16) // 4,), float("nan"), dtype=torch.float32, device="cuda")
    B.osrc_gemm_bf16(A, Bm, Cw, err, ws=ws)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    ref = (A.double() @ Bm.double().T).float()
    assert torch.isfinite(C).all()
    assert float((C - ref).abs().max() / ref.abs().max()) < 1e-5
    if wide:
        assert torch.isnan(Cw[:, N:]).all()
    C2 = C.clone()
    B.osrc_gemm_bf16(A, Bm, Cw, err, ws=ws)
    torch.cuda.synchronize()
    assert torch.equal(C, C2)
