"""The dense basis across batch sizes: the transform of a row, and with it
the row's codes and scale, is one float32 chain over K whatever other rows
the call has, whatever their number, and under a cap on the GEMM's CTA pairs."""

import numpy as np
import pytest
import torch

from paper_2606_04945_gb300 import inputs
from tests import helpers as H
from tests.test_gpu_dense import basis

pytestmark = pytest.mark.gpu

a256 = lambda x: (x + 255) // 256 * 256


@pytest.mark.parametrize("K,dtype", [(1024, "bf16"), (4096, "f16")])
def test_codes_do_not_depend_on_the_batch(abi, K, dtype):
    case = inputs.random_linear(K + 9, 300, K, 128, dtype=dtype, hb=1)
    xf = case.xf
    _, Pt = basis(K, K + 2)
    X, mask = H.dev(case.X, H.torch_dtype(dtype)), H.dev(case.mask)
    a_m, a_u = H.dev(xf.a_m), H.dev(xf.a_u)

    def quantise(L, pairs):
        Xq = torch.empty(L, K // 2, dtype=torch.uint8, device="cuda")
        s_a = torch.empty(L, dtype=torch.float32, device="cuda")
        prev = abi.set_gemm_pair_limit(pairs)
        try:
            ws = abi.sgat_quantize_act_dense(X[:L].contiguous(), mask[:L].contiguous(), a_m, a_u, Pt, xf.d_sh, xf.d_m,
                                             xf.d_u, Xq, s_a)
        finally:
            abi.set_gemm_pair_limit(prev)
        V = ws[a256(L * K * 2): a256(L * K * 2) + 2 * L * K].view(torch.float16).view(L, K)
        return V, Xq, s_a

    all_rows = quantise(300, 0)
    for L in (1, 17, 64, 65, 256, 257):
        for pairs in (0, 8):
            for got, ref in zip(quantise(L, pairs), all_rows):
                assert torch.equal(got, ref[:L]), (L, pairs)
    abi.check_status()


def test_weight_codes_do_not_depend_on_the_batch(abi):
    N, K = 300, 2048
    case = inputs.random_linear(N, 8, K, N + 20, dtype="f16", hb=1)
    _, Pt = basis(K, K + 3)
    W, inv = H.dev(case.W, torch.float16), H.dev(case.xf.inv_a_w)
    out = []
    for n in (N, 64):
        Wq = torch.empty(n, K // 2, dtype=torch.uint8, device="cuda")
        s_w = torch.empty(n, dtype=torch.float32, device="cuda")
        ws = abi.sgat_prepare_weight_dense(W[:n].contiguous(), inv, Pt, Wq, s_w)
        out.append((ws[a256(n * K * 2): a256(n * K * 2) + 2 * n * K].view(torch.float16).view(n, K), Wq, s_w))
    abi.check_status()
    for got, ref in zip(out[1], out[0]):
        assert torch.equal(got, ref[:64])
