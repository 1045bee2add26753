"""The row quantiser's layouts (rows of 1024 features and more) against the
oracle, bit for bit: every Hadamard block size class (stages in layout 1
only, up to layout 2, back in layout 1, layout 3), slices with missing or half
chunks, clusters of slices, gate boundaries inside a group of four, no
smoothing vectors, and the 8-bit codes."""

import numpy as np
import pytest
import torch

from oracle import sgat as osg
from paper_2606_04945_gb300 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu

CASES = [  # K, hb, dtype
    (1024, 1, "f16"), (1536, 2, "bf16"), (1024, 4, "f32"), (2560, 8, "f16"), (1024, 64, "bf16"), (1536, 128, "f16"),
    (3584, 256, "f32"), (4608, 512, "bf16"), (5120, 1024, "f16"), (3072, 1024, "f32"), (2048, 2048, "bf16"),
    (6144, 2048, "f16"), (8192, 4096, "f32"), (20480, 4096, "f16"), (18944, 512, "f16"), (12800, 512, "f32"),
]


@pytest.mark.parametrize("K,hb,dtype", CASES)
@pytest.mark.parametrize("bits", [4, 8])
def test_rows_bitexact(abi, K, hb, dtype, bits):
    L = 5
    rng = np.random.default_rng(K + hb + bits)
    case = inputs.random_linear(K + hb, L, K, 32, dtype="f16" if dtype == "f32" else dtype, hb=hb)
    xf = case.xf
    d_m, d_u = int(rng.integers(1, K // 3)), int(rng.integers(1, K // 3))     # boundaries anywhere
    d_sh = K - d_m - d_u
    smooth = bits == 4
    X = H.dev(case.X, H.torch_dtype(dtype))
    Xq = torch.empty(L, K if bits == 8 else K // 2, dtype=torch.uint8, device="cuda")
    Xe = torch.empty(L, 2 * K if bits == 8 else K, dtype=torch.uint8, device="cuda")
    s_a = torch.empty(L, dtype=torch.float32, device="cuda")
    v = torch.empty(L, K, dtype=torch.float32, device="cuda")
    a_m, a_u = (xf.a_m, xf.a_u) if smooth else (None, None)
    dv = lambda a: None if a is None else H.dev(a)
    abi.sgat_quantize_act(X, H.dev(case.mask), dv(a_m), dv(a_u), hb, d_sh, d_m, d_u, Xq, s_a, bits=bits, Xe=Xe, v_dbg=v)
    torch.cuda.synchronize()
    V = osg.sgat_transform(case.X, case.mask, a_m, a_u, hb, d_sh, d_m, d_u)
    codes, s = osg.sgat_quantize_act(case.X, case.mask, a_m, a_u, hb, d_sh, d_m, d_u, bits)
    assert np.array_equal(v.cpu().numpy(), V)
    assert np.array_equal(s_a.cpu().numpy(), s)
    if bits == 4:
        assert np.array_equal(H.unpack(Xq), codes)
        value = Xe.view(torch.float8_e4m3fn).float().cpu().numpy()
    else:
        assert np.array_equal(Xq.cpu().numpy().view(np.int8), codes)
        value = Xe.view(torch.float16).float().cpu().numpy()
    assert np.array_equal(value, codes.astype(np.float32))


# the compiled-in blocks in the asymmetric mode: one wave and several (whole
# slices only), rows of one CTA and of clusters, half chunks
@pytest.mark.parametrize("L,K,hb,dtype", [(3, 4096, 4096, "f32"), (1100, 4096, 4096, "f16"), (1300, 4096, 4096, "bf16"),
                                          (6, 3584, 512, "bf16"), (5, 7680, 512, "f16"), (7, 4608, 512, "f32"),
                                          (6, 1024, 1024, "f16"), (5, 7168, 1024, "bf16"), (6, 2048, 2048, "f16"),
                                          (5, 6144, 2048, "bf16"), (4, 1536, 256, "f16")])
def test_rows_asym_bitexact(abi, L, K, hb, dtype):
    case = inputs.random_linear(K + L, L, K, 32, dtype="f16" if dtype == "f32" else dtype, hb=hb)
    xf = case.xf
    X = H.dev(case.X, H.torch_dtype(dtype))
    Xq = torch.empty(L, K // 2, dtype=torch.uint8, device="cuda")
    Xe = torch.empty(L, K + 128, dtype=torch.uint8, device="cuda")
    s_a = torch.empty(L, dtype=torch.float32, device="cuda")
    z_a = torch.empty(L, dtype=torch.int32, device="cuda")
    abi.sgat_quantize_act_asym(X, H.dev(case.mask), H.dev(xf.a_m), H.dev(xf.a_u), hb, xf.d_sh, xf.d_m, xf.d_u, Xq, s_a,
                               z_a, Xe=Xe)
    torch.cuda.synchronize()
    codes, s, z = osg.sgat_quantize_act_asym(case.X, case.mask, xf.a_m, xf.a_u, hb, xf.d_sh, xf.d_m, xf.d_u)
    nibbles = Xq.cpu().numpy()
    assert np.array_equal(np.stack([nibbles & 15, nibbles >> 4], -1).reshape(L, K), codes)
    assert np.array_equal(Xe[:, :K].view(torch.float8_e4m3fn).float().cpu().numpy(), codes.astype(np.float32))
    assert np.array_equal(s_a.cpu().numpy(), s)
    assert np.array_equal(z_a.cpu().numpy(), z)


@pytest.mark.parametrize("K,hb", [(1024, 1), (2048, 2048), (4096, 1)])
def test_rows_nibbles_saturate(abi, K, hb):
    """Packed codes of rows without a finite reciprocal scale saturate: with
    amax <= 7 / FLT_MAX the reciprocal 7 / amax is infinite, so every product
    is +-inf and its code the end of the nibble's range on that side; an
    infinite element has the reciprocal 0, the product inf * 0 (no number) and
    the code 7, the row's finite elements 0."""
    L = 2
    X = np.zeros((L, K), np.float32)
    X[0] = np.where(np.arange(K) % 3 == 0, 1e-38, -1e-38) if hb == 1 else 0
    if hb == 1:
        X[1] = 1.0
        X[1, 5] = np.inf
    else:
        X[0, 0] = 1e-38                                    # its transform: 1e-38 in every element of the block
    mask = np.zeros(L, np.uint8)
    Xq = torch.empty(L, K // 2, dtype=torch.uint8, device="cuda")
    s_a = torch.empty(L, dtype=torch.float32, device="cuda")
    abi.sgat_quantize_act(H.dev(X), H.dev(mask), None, None, hb, K, 0, 0, Xq, s_a)
    codes = H.unpack(Xq)
    assert np.array_equal(codes[0], np.where(X[0] < 0, -8, 7) if hb == 1 else np.full(K, 7))
    if hb == 1:
        assert codes[1, 5] == 7 and not np.any(np.delete(codes[1], 5))
