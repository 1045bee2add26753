"""The few-token W4A4 GEMM (operands swapped, K split over a cluster) against
the oracle: integer accumulators exact, outputs within the dequantisation
bound, at the edges of its token tiles, splits of K that do not divide it,
channel counts that are no multiple of the tile, the largest sums, and the
SwiGLU epilogue against the pair kernel (selected by a cap on its pairs)."""

import numpy as np
import pytest
import torch

from oracle import sgat as osg
from paper_2606_04945_gb300 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu


def _gemm(abi, qa, qw, s_a, s_w, out, bias):
    L, N = qa.shape[0], qw.shape[0]
    Y = torch.empty(L, N, dtype=H.torch_dtype(out), device="cuda")
    acc = torch.empty(L, N, dtype=torch.int32, device="cuda")
    abi.w4a4_gemm(None, H.dev(s_a), None, H.dev(s_w), Y, bias=None if bias is None else H.dev(bias), acc_dbg=acc,
                  Xe=H.dev(H.e4m3_bytes(qa)), We=H.dev(H.e4m3_bytes(qw)))
    abi.check_status()
    return Y, acc.cpu().numpy()


# L around the token tiles (16, 32, 64, 128), split 8 of 9 and 5 K blocks, one part per tile
# (19 x 1024 over 40000 channels), ragged channels (32, 160, 4128)
@pytest.mark.parametrize("L,N,K,out,bias", [(1, 1024, 2048, "f16", False), (16, 160, 1152, "bf16", True),
                                            (17, 4128, 640, "f32", False), (32, 4096, 4096, "f16", True),
                                            (33, 32, 4096, "f16", False), (64, 512, 2176, "f32", True),
                                            (65, 1024, 8192, "bf16", False), (128, 2048, 12288, "f16", False),
                                            (200, 1024, 12288, "f16", True), (19, 40000, 1024, "f16", False)])
def test_few_tokens_exact(abi, L, N, K, out, bias):
    qa, qw, s_a, s_w = H.gemm_codes(L + N + K, L, N, K)
    b = np.random.default_rng(L).normal(0, 0.1, N).astype(np.float32) if bias else None
    Y, acc = _gemm(abi, qa, qw, s_a, s_w, out, b)
    bn, split = abi.last_gemm_tile()
    assert bn == 128 and 1 <= split <= 8, (bn, split)
    ref = osg.int_gemm(qa, qw)
    assert np.array_equal(acc, ref)
    prev = abi.set_gemm_pair_limit(10 ** 6)            # the pair kernel: the same bits
    try:
        Y2, acc2 = _gemm(abi, qa, qw, s_a, s_w, out, b)
    finally:
        abi.set_gemm_pair_limit(prev)
    assert abi.last_gemm_tile()[0] in (224, 256)
    assert torch.equal(Y, Y2) and np.array_equal(acc, acc2)
    if not (bias and out == "f32"):                    # (a bias can cancel the product: only the bits above bind)
        H.assert_output_close(H.host(Y), osg.dequant(ref, s_a, s_w, b), out)


def test_few_tokens_largest_sums(abi):
    """|acc| = 49 K at K = 65536, split over eight parts: exact in float32."""
    L, N, K = 24, 256, 65536
    qa, qw = np.full((L, K), 7, np.int32), np.full((N, K), -7, np.int32)
    qw[1::2] *= -1
    one = lambda n: np.ones(n, np.float32)
    _, acc = _gemm(abi, qa, qw, one(L), one(N), "f32", None)
    assert abi.last_gemm_tile()[0] == 128
    assert np.array_equal(acc, np.broadcast_to(np.where(np.arange(N) % 2 == 1, 49 * K, -49 * K), (L, N)))


@pytest.mark.parametrize("L,K,F,dtype", [(32, 4096, 2048, "f16"), (5, 1024, 496, "bf16"), (100, 8192, 512, "f16")])
def test_few_tokens_swiglu(abi, L, K, F, dtype):
    case = inputs.random_linear(L + K + F, L, K, 2 * F, dtype=dtype, bias=True)
    xf, td = case.xf, H.torch_dtype(dtype)
    Wq = torch.empty(2 * F, K // 2, dtype=torch.uint8, device="cuda")
    s_w = torch.empty(2 * F, dtype=torch.float32, device="cuda")
    abi.sgat_prepare_weight(H.dev(case.W, td), H.dev(xf.inv_a_w), xf.hb, Wq, s_w)
    We = torch.empty(2 * F, K, dtype=torch.uint8, device="cuda")
    abi.w4_unpack_e4m3(Wq, We)
    ws = torch.empty(abi.sgat_linear_workspace_size(L, K, False), dtype=torch.uint8, device="cuda")
    args = (H.dev(case.X, td), H.dev(case.mask), H.dev(xf.a_m), H.dev(xf.a_u), xf.hb, xf.d_sh, xf.d_m, xf.d_u, Wq, s_w)
    out = []
    for limit in (0, 10 ** 6):
        prev = abi.set_gemm_pair_limit(limit)
        try:
            Hb = torch.empty(L, F, dtype=td, device="cuda")
            abi.sgat_linear_swiglu(*args, Hb, ws, bias=H.dev(case.bias), We=We)
            abi.check_status()
        finally:
            abi.set_gemm_pair_limit(prev)
        assert (abi.last_gemm_tile()[0] == 128) == (limit == 0)
        out.append(Hb)
    assert torch.equal(out[0], out[1])


# 8-bit codes held as fp16: one accumulator per part (16 stages of 64 K), two, a part that ends
# inside its second one, the largest magnitudes, and one part per tile
@pytest.mark.parametrize("L,N,K,out,extreme", [(1, 128, 128, "f16", False), (32, 512, 4096, "bf16", False),
                                               (17, 1024, 12288, "f16", True), (70, 256, 8320, "f32", False),
                                               (128, 4096, 4096, "f16", False), (9, 40960, 1024, "f16", True)])
def test_few_tokens_8bit_exact(abi, L, N, K, out, extreme):
    rng = np.random.default_rng(L + N + K)
    draw = (lambda r: np.full((r, K), 127) * rng.choice([-1, 1], (r, 1))) if extreme else \
        (lambda r: rng.integers(-127, 128, (r, K)))
    qa, qw = draw(L).astype(np.int64), draw(N).astype(np.int64)
    s_a, s_w = rng.uniform(0.01, 1, L).astype(np.float32), rng.uniform(0.01, 1, N).astype(np.float32)
    bias = rng.normal(0, 0.1, N).astype(np.float32) if L == 32 else None
    Xe, We = H.dev(qa.astype(np.float16)), H.dev(qw.astype(np.float16))
    res = []
    for limit in (0, 10 ** 6):
        prev = abi.set_gemm_pair_limit(limit)
        try:
            Y = torch.empty(L, N, dtype=H.torch_dtype(out), device="cuda")
            acc = torch.empty(L, N, dtype=torch.int32, device="cuda")
            abi.w8a8_gemm(Xe, H.dev(s_a), We, H.dev(s_w), Y, bias=None if bias is None else H.dev(bias), acc_dbg=acc)
            abi.check_status()
        finally:
            abi.set_gemm_pair_limit(prev)
        assert (abi.last_gemm_tile()[0] == 128) == (limit == 0)
        res.append((Y, acc))
    ref = (qa.astype(np.float64) @ qw.T.astype(np.float64)).astype(np.int64)       # exact below 2^53
    assert np.array_equal(res[0][1].cpu().numpy(), ref)
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])


@pytest.mark.parametrize("L,N,K,dt", [(1, 32, 64, "f16"), (20, 4096, 4096, "f16"), (33, 160, 2112, "bf16"),
                                      (100, 1024, 8192, "bf16"), (64, 512, 16384, "f16")])
def test_few_tokens_16bit(abi, L, N, K, dt):
    """Plain 16-bit product: float32 sums of K / split terms and their sum over
    at most eight parts stay within the bound of one chain of K, and the error
    against float64 is no larger than the pair kernel's (5 % for the draw)."""
    rng = np.random.default_rng(L + N + K)
    rnd = (lambda x: x.astype(np.float16).astype(np.float32)) if dt == "f16" else inputs.round_to_bf16
    A, B = (rnd(rng.standard_normal((r, K)).astype(np.float32)) for r in (L, N))
    ref = A.astype(np.float64) @ B.astype(np.float64).T
    mag = np.abs(A).astype(np.float64) @ np.abs(B).astype(np.float64).T
    err = []
    for limit in (0, 10 ** 6):
        prev = abi.set_gemm_pair_limit(limit)
        try:
            C = torch.empty(L, N, dtype=H.torch_dtype(dt), device="cuda")
            abi.fp16_gemm_ref(H.dev(A, H.torch_dtype(dt)), H.dev(B, H.torch_dtype(dt)), C)
            abi.check_status()
        finally:
            abi.set_gemm_pair_limit(prev)
        assert (abi.last_gemm_tile()[0] == 128) == (limit == 0)
        got = H.host(C).astype(np.float64)
        tol = np.maximum(H.half_spacing(ref, dt), 2.0 ** -11 * np.abs(ref) if dt == "f16" else 0) + 2.0 ** -22 * np.sqrt(K) * mag
        assert np.all(np.abs(got - ref) <= tol)
        err.append(np.linalg.norm(got - ref))
    assert err[0] <= 1.05 * err[1]
