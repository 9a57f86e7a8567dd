"""cfr_gemm_bf16 where its tiles begin and end, and the leaf rows read back after iterations that
compute one player's outputs at a time."""
import numpy as np
import pytest

from oracle import leafnet as ln
from paper_2605_19928_gb300 import capi, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_19928_gb300 import build as pbuild
    pbuild.build()
    capi.load()


# rows around the 128- and 256-row halves of a tile; column counts whose widest tiles are 128, 192, 160,
# 224 and 256; one, few and many 64-wide steps of K; enough rows for several tiles a pair (wide and
# narrow tiles), the last one ragged
@pytest.mark.parametrize("M,N,K", [(1, 128, 64), (127, 128, 128), (129, 384, 192), (256, 640, 576), (257, 2688, 64),
                                   (624, 512, 2752), (5001, 2688, 128), (20001, 512, 192), (40005, 512, 64)])
@pytest.mark.parametrize("act,out_f32,with_bias", [(False, True, True), (True, True, False), (True, False, True),
                                                   (False, False, False)])
def test_edges_match_fp64(M, N, K, act, out_f32, with_bias):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)
    B = (torch.randn(N, K, device="cuda", generator=g) / K ** 0.5).to(torch.bfloat16)
    bias = torch.randn(N, device="cuda", generator=g) if with_bias else None
    buf = torch.full((M + 256, N), 7.0, dtype=torch.float32 if out_f32 else torch.bfloat16, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    capi.cfr_gemm_bf16(A, B, bias, buf[:M], act, err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert bool((buf[M:] == 7.0).all())  # nothing past the last row
    want = A.double() @ B.double().T
    terms = A.double().abs() @ B.double().abs().T
    if bias is not None:
        want += bias.double()
        terms += bias.double().abs()
    tol = 2e-6 * (terms + want.abs()) + 1e-30  # FP32 accumulation and the bias
    if act:
        want = torch.nn.functional.gelu(want)
        tol = 1.13 * tol + 1e-6 * terms  # through GELU's slope; its own FP32 steps
    if not out_f32:
        tol = tol + want.abs() * 2.0 ** -8 * (1 + 2.0 ** -7) + 1e-38  # one rounding to BF16
    assert bool(((buf[:M].double() - want).abs() <= tol).all())


@pytest.mark.parametrize("alternating", [True, False])
def test_leaf_outputs_of_both_players_are_read_after_iterations(alternating):
    from paper_2605_19928_gb300 import leafnet_train
    spec = synth.turn_subgame(n_hands=200, seed=3, range_seed=4, bet_sizes=(1.0, synth.ALL_IN), max_raises=2)
    spec.depth_limit = 1
    W, b = leafnet_train.load_weights()
    tree = capi.cfr_tree_create(spec, capi.make_opts("dcfr", precision="single", alternating=alternating))
    try:
        capi.cfr_set_leaf_net(tree, W, b)
        capi.cfr_iterate(tree, 3)
        _, _, row0 = capi.cfr_leaf_info(tree)[-1]
        X = ln.bf16_from_bits(capi.cfr_read_leaf_rows(tree, 0, row0, 48))
        Y = capi.cfr_read_leaf_rows(tree, 1, row0, 48)
        want = ln.forward(X, list(zip([ln.bf16_from_bits(w) for w in W], b)))
        scale = np.max(np.abs(want), axis=1, keepdims=True)
        assert np.max(np.abs(Y - want) / scale) <= 3e-2  # hidden activations round to BF16 on both sides
    finally:
        capi.cfr_tree_destroy(tree)
