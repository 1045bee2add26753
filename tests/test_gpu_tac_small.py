"""TAC for blocks of up to 32 (CUDA cores, tiles of 128 channels x 64 tokens, 128
for blocks of 32; a thread takes two tokens half a tile apart) against float32
sums in the kernel's order (ascending inputs, fused multiply-add, then + d): bit
for bit but for double roundings of the reference, at the edges of its tiles."""

import numpy as np
import pytest
import torch

from paper_2606_04945_gb300 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g,L,C,zin,zout,with_d", [(4, 1, 8, "f16", "f16", True), (4, 130, 4096, "bf16", "f32", True),
                                                  (8, 127, 136, "f16", "bf16", False), (8, 128, 128, "f32", "f16", True),
                                                  (16, 129, 272, "f16", "f16", True), (16, 300, 2560, "bf16", "bf16", False),
                                                  (32, 64, 96, "f32", "f32", True), (32, 257, 160, "f16", "f16", True),
                                                  # one tile of 64 tokens: its halves' edges, its last token, one more
                                                  (4, 31, 136, "f16", "f16", True), (8, 32, 128, "bf16", "f32", True),
                                                  (16, 33, 272, "f16", "f16", False), (4, 63, 8, "f32", "f32", True),
                                                  (8, 64, 264, "f16", "f16", True), (16, 65, 128, "bf16", "bf16", True),
                                                  (8, 63, 128, "f16", "f16", True), (16, 64, 48, "f16", "f32", True),
                                                  (4, 65, 128, "f16", "bf16", True)])
def test_tac_small_blocks(abi, g, L, C, zin, zout, with_d):
    rng = np.random.default_rng(g + L + C)
    Z = rng.standard_normal((L, C)).astype(np.float32)
    Z = Z.astype(np.float16).astype(np.float32) if zin == "f16" else (inputs.round_to_bf16(Z) if zin == "bf16" else Z)
    tp = inputs.make_tac(rng, C, g, noise=0.5)
    out = torch.full((L, C), float("nan"), dtype=H.torch_dtype(zout), device="cuda")
    abi.tac_apply(H.dev(Z, H.torch_dtype(zin)), H.dev(tp.M), H.dev(tp.d) if with_d else None, g, out)
    abi.check_status()
    # a fused multiply-add of float32 values in float64: the product is exact, and
    # the sum's second rounding (to float32) differs from the single one only
    # where the float64 sum lies next to a rounding boundary
    z, M = Z.reshape(L, C // g, g).astype(np.float64), tp.M.astype(np.float64)
    acc = np.zeros((L, C // g, g))
    for j in range(g):
        acc = (z[:, :, j, None] * M[None, :, :, j] + acc).astype(np.float32).astype(np.float64)
    ref = (acc + tp.d.astype(np.float64)[None] if with_d else acc).astype(np.float32).reshape(L, C)
    got = H.host(out)
    if zout == "f32":
        assert np.mean(got != ref) < 1e-5 and np.all(np.abs(got - ref) <= 2.0 ** -22 * (np.abs(ref) + 1))
    else:
        rnd = ref.astype(np.float16).astype(np.float32) if zout == "f16" else inputs.round_to_bf16(ref)
        assert np.mean(got != rnd) < 1e-5 and np.all(np.abs(got - rnd) <= 2.0 ** -7 * (np.abs(rnd) + 2.0 ** -14))
