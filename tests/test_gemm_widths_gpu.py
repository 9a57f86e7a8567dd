"""cfr_gemm_bf16 gives a row the same bits whatever the number of rows, and so the tile width, the
epilogue's warps and the rounds of tiles; and those are right against FP64 with several rounds a pair."""
import pytest

from paper_2605_19928_gb300 import capi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_19928_gb300 import build as pbuild
    pbuild.build()
    capi.load()


@pytest.mark.parametrize("N,K", [(512, 64), (512, 1024), (384, 2752), (2688, 512), (128, 512)])
@pytest.mark.parametrize("act,out_f32", [(False, True), (True, True), (True, False), (False, False)])
def test_rows_keep_their_bits_at_every_row_count(N, K, act, out_f32):
    import torch
    M = 20005  # three rounds of the widest tiles and more, the last ragged
    g = torch.Generator(device="cuda").manual_seed(N + K)
    A = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)
    B = (torch.randn(N, K, device="cuda", generator=g) / K ** 0.5).to(torch.bfloat16)
    bias = torch.randn(N, device="cuda", generator=g)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = {}
    for m in (M, 5003, 700, 65, 1):
        out[m] = torch.full((m, N), 7.0, dtype=torch.float32 if out_f32 else torch.bfloat16, device="cuda")
        capi.cfr_gemm_bf16(A[:m], B, bias, out[m], act, err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    for m, c in out.items():
        assert torch.equal(c, out[M][:m]), m
    rows = slice(M - 600, M)  # the last rounds
    want = A[rows].double() @ B.double().T + bias.double()
    terms = A[rows].double().abs() @ B.double().abs().T + bias.double().abs()
    tol = 2e-6 * (terms + want.abs()) + 1e-30  # FP32 accumulation and the bias
    if act:
        want = torch.nn.functional.gelu(want)
        tol = 1.13 * tol + 1e-6 * terms  # through GELU's slope; its own FP32 steps
    if not out_f32:
        tol = tol + want.abs() * 2.0 ** -8 * (1 + 2.0 ** -7) + 1e-38  # one rounding to BF16
    assert bool(((out[M][rows].double() - want).abs() <= tol).all())
