"""The attention kernel's S buffers across work items: pass 1 goes round three
(the third lies in the accumulator's columns, handed over by each item's
epilogue), pass 2 round two. One to five key chunks, several items per CTA,
against the same heads computed alone (one item per CTA), bit for bit; and a
model of the buffers' parity waits."""

import pytest
import torch

D = 128


@pytest.mark.gpu
@pytest.mark.parametrize("L", [128, 256, 384, 512, 640])
def test_items_per_cta(abi, L):
    nq, sms = L // D, torch.cuda.get_device_properties(0).multi_processor_count
    Hh = 3 * sms // nq + 1                                   # more than three items for some CTAs
    C = Hh * D
    g = torch.Generator(device="cuda").manual_seed(L)
    qkv = torch.randn(L, 3 * C, device="cuda", generator=g).half()
    M = (torch.eye(D, device="cuda") + 0.05 * torch.randn(Hh, D, D, device="cuda", generator=g)).contiguous()
    d = torch.randn(Hh, D, device="cuda", generator=g)
    q, k, v = qkv[:, :C], qkv[:, C:2 * C], qkv[:, 2 * C:]

    def attention(h0, n):
        Mp = torch.empty(abi.tac_prepared_bytes(D * n, D), dtype=torch.uint8, device="cuda")
        abi.tac_prepare(M[h0:h0 + n].contiguous(), D, torch.float16, Mp)
        ws = torch.empty(abi.attention_pv_tac_workspace_size(L, n), dtype=torch.uint8, device="cuda")
        Z = torch.empty(L, n * D, dtype=torch.float16, device="cuda")
        s = slice(h0 * D, (h0 + n) * D)
        abi.attention_pv_tac(q[:, s], k[:, s], v[:, s], n, Mp, d[h0:h0 + n].contiguous(), Z, workspace=ws)
        return Z
    Z = attention(0, Hh)
    step = max(1, sms // nq // 2)                            # heads whose items all fit the SMs at once
    parts = [attention(h0, min(step, Hh - h0)) for h0 in range(0, Hh, step)]
    abi.check_status()
    assert torch.isfinite(Z.float()).all() and float(Z.float().std()) > 0
    assert torch.equal(Z, torch.cat(parts, 1))


@pytest.mark.parametrize("nk", [1, 2, 3, 4, 5, 6, 7, 64])
def test_buffer_parities(nk):
    """The masks of both sides (one bit per buffer) against counted phases:
    every wait names the phase it means, and the barrier is at most one phase
    on. The MMA warp runs as far ahead as its waits let it."""
    full, empty = [0, 0, 0], [0, 0, 0]                       # completed phases
    mma_uses, soft_uses = 0, 0
    counted = [0, 0, 0]                                      # phases of s_empty the MMA warp has accounted for
    reads = []                                               # scores waiting for the softmax warps: buffer, kind

    def passes(phases, parity):                              # a parity wait: the phase of that parity has completed
        return (phases & 1) != parity

    def softmax_step():
        nonlocal soft_uses
        b = reads.pop(0)
        assert passes(full[b], soft_uses >> b & 1)
        soft_uses ^= 1 << b
        empty[b] += 1

    def wait_empty(b, parity, want):
        while empty[b] < want:
            assert reads, "deadlock"
            softmax_step()
        assert empty[b] == want and passes(empty[b], parity)

    def qk(b):
        nonlocal mma_uses
        wait_empty(b, (mma_uses >> b & 1) ^ 1, counted[b])
        full[b] += 1
        reads.append(b)
        mma_uses ^= 1 << b
        counted[b] += 1
    for item in range(4):
        for it in range(nk):
            qk(it % 3)
        mma_uses ^= 4                                        # the release of the TAC accumulator
        counted[2] += 1
        for j in range(min(2, nk)):
            qk(j)
        for j in range(nk):
            b = j & 1
            wait_empty(b, (mma_uses >> b & 1) ^ 1, counted[b])       # P(j) in place
            if j == 0:                                       # P V^T(0) overwrites the third buffer
                assert 2 not in reads
            if j + 2 < nk:
                qk(b)
        assert not reads
        empty[2] += 1                                        # the epilogue has read the TAC accumulator
