"""The attention's V quantiser (codes and channel scales in the workspace)
against the oracle, bit for bit, at key counts that leave a cluster's last CTA
with fewer chunks and at every number of chunks per CTA, with an all-zero
channel and a channel of one sign."""

import numpy as np
import pytest
import torch

from oracle import attention as oatt
from paper_2606_04945_gb300 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu
D = 128


@pytest.mark.parametrize("L,Hkv,dt", [(128, 1, "f16"), (896, 3, "bf16"), (1152, 1, "bf16"), (2944, 2, "f16"),
                                      (4096, 1, "bf16"), (4224, 1, "f16"), (8192, 1, "bf16")])
def test_v_codes(abi, L, Hkv, dt):
    rng = np.random.default_rng(L + Hkv)
    C = D * Hkv
    V = rng.standard_normal((L, C)).astype(np.float32) * rng.uniform(0.1, 30, C).astype(np.float32)
    V[:, 5] = 0
    V[:, 77] = np.abs(V[:, 77])
    V = V.astype(np.float16).astype(np.float32) if dt == "f16" else inputs.round_to_bf16(V)
    td = H.torch_dtype(dt)
    QKV = torch.zeros(L, 3 * C, dtype=td, device="cuda")
    QKV[:, 2 * C:] = H.dev(V, td)
    Mp = torch.empty(abi.tac_prepared_bytes(C, D), dtype=torch.uint8, device="cuda")
    abi.tac_prepare(torch.eye(D, device="cuda").repeat(Hkv, 1, 1).contiguous(), D, torch.float16, Mp)
    ws = torch.full((abi.attention_pv_tac_workspace_size(L, Hkv),), 0xEE, dtype=torch.uint8, device="cuda")
    Z = torch.empty(L, C, dtype=td, device="cuda")
    abi.attention_pv_tac(QKV[:, :C], QKV[:, C:2 * C], QKV[:, 2 * C:], Hkv, Mp, None, Z, workspace=ws)
    abi.check_status()
    codes, t = oatt.v_codes(V)
    n = C * L * 2
    got = ws[:n].view(torch.float16).view(C, L).float().cpu().numpy()
    off = (n + 255) // 256 * 256
    assert np.array_equal(got.T, codes.astype(np.float32))
    assert np.array_equal(ws[off:off + 4 * C].view(torch.float32).cpu().numpy(), t)
