"""The work that a user of this library has it do, case by case.

A case is one call (or one captured step) through the public entry points: the
SGAT linear in its code widths and bases, the attention-projection and MLP
steps, the quantised attention product, TAC, weight preparation, and the two
whole models of the package (the LLaDA-shaped denoising stack and the
Dream-shaped block). Sizes are those of the package's own workloads
(``inputs.py``, ``stack.py``), with small and ragged token counts between
them, as batches of a denoising server have them.

``listed()`` names the cases; ``draw(rng)`` gives another one of the same
ranges. ``prepare`` builds what a program holds before the call, ``run`` is
one pass, ``exact`` is the same computation in float64 torch.
"""

import math

import numpy as np
import torch

from paper_2606_04945_gb300 import abi, inputs
from paper_2606_04945_gb300.dream import DreamBlock
from paper_2606_04945_gb300.pipeline import AttentionProjections
from paper_2606_04945_gb300.stack import DenoiseStack, StackConfig

DTYPE = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
DEV = "cuda"


def listed():
    return [
        # one small linear with TAC (256 tokens x 512): launch and latency
        dict(name="linear_256x512_tac64", kind="linear", scheme="w4", L=256, K=512, N=512, dtype="f16", tac=64,
             bias=False),
        # one block of 32 tokens of semi-autoregressive decoding through the
        # LLaDA QKV projection: the weights are read for few rows
        dict(name="linear_block32_qkv", kind="linear", scheme="w4", L=32, K=4096, N=12288, dtype="f16", tac=0,
             bias=False),
        # the W8A8 setting, an O projection on a ragged batch
        dict(name="linear_w8a8_1000", kind="linear", scheme="w8", L=1000, K=4096, N=4096, dtype="bf16", tac=0,
             bias=True),
        # a learned dense basis in place of the Hadamard transform, ragged
        dict(name="linear_dense_777", kind="linear", scheme="dense", L=777, K=4096, N=4096, dtype="f16", tac=0,
             bias=False),
        # the attention projections of one LLaDA denoising step (QKV of X, TAC
        # + O of Z), replayed from its captured graph
        dict(name="attn_step_1024", kind="attn_step", L=1024),
        # the LLaDA MLP of one step: gate + up with SwiGLU, then down
        dict(name="mlp_1024", kind="mlp", L=1024, H=4096, F=12288, dtype="f16"),
        # quantised softmax-value product with TAC: LLaDA heads, fp16
        dict(name="attention_1024_h32", kind="attention", L=1024, H=32, Hkv=32, dtype="f16"),
        # the same with grouped key/value heads, bf16 (one Dream sequence)
        dict(name="attention_2048_gqa", kind="attention", L=2048, H=28, Hkv=4, dtype="bf16"),
        # TAC alone over a large batch
        dict(name="tac_8192x4096", kind="tac", L=8192, C=4096, g=128, dtype="f16", out="f16", prepared=True),
        # weight preparation of the LLaDA gate + up projection
        dict(name="prepare_24576x4096", kind="weights", N=24576, K=4096, dtype="f16"),
        # one denoising step of the whole LLaDA-shaped stack, captured
        dict(name="stack_step_1024", kind="stack", seq=1024, layers=4, step=31),
        # one pass of the Dream-shaped block, 4 x 2048 tokens, captured
        dict(name="dream_block_4x2048", kind="dream", batch=4, seq=2048),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng):
    """A feature count: a model's width, or another multiple of 128."""
    if rng.random() < 0.6:
        return rng.choice([512, 1024, 2048, 3584, 4096, 4096, 12288])
    return 128 * _log_int(rng, 2, 64)


def draw(rng):
    u = rng.random()
    if u < 0.5:
        scheme = rng.choice(["w4", "w4", "w4", "w8", "asym", "dense"])
        K = _width(rng)
        if scheme in ("asym", "dense"):
            K = min(K, 4096)
        N = 128 * _log_int(rng, 4, 192) if scheme == "w8" else 32 * _log_int(rng, 16, 768)
        L = _log_int(rng, 1, 8192)
        L = max(1, min(L, int(1e12 / (2.0 * N * K))))
        tac = rng.choice([0, 0, 0, 64, 128]) if scheme in ("w4", "w8") and K % 128 == 0 else 0
        return dict(kind="linear", scheme=scheme, L=L, K=K, N=N, dtype=rng.choice(["f16", "bf16"]), tac=tac,
                    bias=rng.random() < 0.4)
    if u < 0.65:
        H, Hkv = rng.choice([(32, 32), (28, 4), (32, 8), (8, 8), (16, 2)])
        return dict(kind="attention", L=128 * _log_int(rng, 1, 32), H=H, Hkv=Hkv, dtype=rng.choice(["f16", "bf16"]))
    if u < 0.77:
        g = rng.choice([16, 64, 64, 128, 128, 128])
        dtype = rng.choice(["f16", "bf16"])
        return dict(kind="tac", L=_log_int(rng, 16, 16384), C=128 * _log_int(rng, 4, 40), g=g, dtype=dtype,
                    out=rng.choice([dtype, dtype, "f32"]), prepared=g >= 64 and rng.random() < 0.8)
    if u < 0.85:
        return dict(kind="weights", N=32 * _log_int(rng, 16, 768), K=_width(rng), dtype=rng.choice(["f16", "bf16"]))
    if u < 0.93:
        H, F = rng.choice([(4096, 12288), (3584, 18944), (2048, 5632)])
        return dict(kind="mlp", L=_log_int(rng, 1, 4096), H=H, F=F, dtype=rng.choice(["f16", "bf16"]))
    if u < 0.97:
        return dict(kind="attn_step", L=_log_int(rng, 16, 4096))
    return dict(kind="stack", seq=128 * rng.randint(3, 8), layers=rng.choice([1, 2, 4]), step=rng.randint(0, 63))


# ---------------------------------------------------------------------------
# Inputs, from the seed alone
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, device=DEV, generator=g)


def _acts(g, L, K, dtype):
    """N(0, 1) activations with 0.5 % of the channels Student-t(3)."""
    X = _randn(g, L, K)
    n = max(1, round(0.005 * K))
    cols = torch.randperm(K, device=DEV, generator=g)[:n]
    X[:, cols] = _randn(g, L, n) / (_randn(g, 3, L, n).square().sum(0) / 3).sqrt()
    return X.to(DTYPE[dtype])


def _weight(g, N, K, dtype):
    return (_randn(g, N, K) * 0.02).to(DTYPE[dtype])


def _mask(L, frac=0.375):
    """The last frac of the tokens still masked."""
    m = torch.zeros(L, dtype=torch.uint8, device=DEV)
    m[L - int(round(frac * L)):] = 1
    return m


def _smoothing(X, mask):
    """Per-state smoothing (a_m, a_u) and the weight side's inverse."""
    out = []
    for state in (1, 0):
        rows = X[mask == state].double().abs()
        if rows.shape[0] == 0:
            out.append(torch.ones(X.shape[1], dtype=torch.float64, device=DEV))
            continue
        a = rows.amax(0).clamp_min(1e-3) ** -0.5
        out.append(a / a.log().mean().exp())
    a_m, a_u = out
    return a_m.float(), a_u.float(), (1.0 / (a_m * a_u).sqrt()).float()


def _tac(g, C, G):
    M = torch.eye(G, device=DEV)[None] + 0.01 * _randn(g, C // G, G, G)
    return M.contiguous(), 0.01 * _randn(g, C // G, G)


def _basis(g, K):
    return torch.linalg.qr(_randn(g, K, K))[0].t().contiguous().half()


def _linear_inputs(g, L, K, N, dtype, scheme="w4", tac=0, bias=False):
    X = _acts(g, L, K, dtype)
    mask = _mask(L)
    a_m, a_u, inv = _smoothing(X, mask)
    d_sh, d_m, d_u = inputs.default_gates(K)
    s = dict(X=X, mask=mask, a_m=a_m, a_u=a_u, inv=inv, W=_weight(g, N, K, dtype), hb=inputs.hadamard_block(K),
             gate=(d_sh, d_m, d_u), scheme=scheme, bias=0.02 * _randn(g, N) if bias else None, M=None, d=None, g=tac)
    if tac:
        s["M"], s["d"] = _tac(g, K, tac)
    if scheme == "dense":
        s["Pt"] = _basis(g, K)
    return s


def _mlp_inputs(case, g):
    L, H, F, dt = case["L"], case["H"], case["F"], case["dtype"]
    gu = _linear_inputs(g, L, H, 2 * F, dt)
    down = _linear_inputs(g, L, F, H, dt)          # its X is the calibration sample of the down projection
    return gu, down


def _attention_inputs(case, g):
    L, H, Hkv, dt = case["L"], case["H"], case["Hkv"], DTYPE[case["dtype"]]
    qkv = _randn(g, L, 128 * (H + 2 * Hkv)).to(dt)
    M, d = _tac(g, 128 * H, 128)
    return qkv, M, d


def _np_linear(s, dtype, tac=None):
    to = lambda t: t.cpu().numpy() if t.dtype != torch.bfloat16 else t.float().cpu().numpy()
    K = s["X"].shape[1]
    d_sh, d_m, d_u = s["gate"]
    xf = inputs.SgatParams(K=K, hb=s["hb"], a_m=to(s["a_m"]), a_u=to(s["a_u"]), inv_a_w=to(s["inv"]), d_sh=d_sh,
                           d_m=d_m, d_u=d_u)
    return inputs.LinearCase("case", to(s["X"]), dtype, to(s["mask"]), to(s["W"]), xf,
                             tac=inputs.TacParams(C=K, g=s["g"], M=to(s["M"]), d=to(s["d"])) if s["g"] else None)


def _dream_case(case, g):
    """A DreamBlockCase from the seed: numpy arrays, as its constructor takes."""
    batch, seq, H, F, heads, kv = case["batch"], case["seq"], 3584, 18944, 28, 4
    L = batch * seq
    t = lambda x: x.float().cpu().numpy()
    one = torch.zeros(seq, dtype=torch.uint8, device=DEV)
    gen_len = min(256, seq)
    mask = []
    for _ in range(batch):          # low-confidence remasking: half of the generated positions still masked
        m = one.clone()
        m[seq - gen_len + torch.randperm(gen_len, device=DEV, generator=g)[: gen_len // 2]] = 1
        mask.append(m)
    mask = torch.cat(mask)
    X = _acts(g, L, H, "bf16")
    nqkv = (heads + 2 * kv) * 128
    W = {n: _weight(g, *sh, "bf16") for n, sh in dict(W_qkv=(nqkv, H), W_o=(H, H), W_gate=(F, H), W_up=(F, H),
                                                    W_down=(H, F)).items()}
    M, d = _tac(g, H, 128)

    def xf(sample, m):
        a_m, a_u, inv = _smoothing(sample, m)
        K = sample.shape[1]
        d_sh, d_m, d_u = inputs.default_gates(K)
        return inputs.SgatParams(K=K, hb=inputs.hadamard_block(K), a_m=t(a_m), a_u=t(a_u), inv_a_w=t(inv), d_sh=d_sh,
                                 d_m=d_m, d_u=d_u)
    calib = lambda K: xf(_acts(g, seq, K, "bf16"), mask[:seq])
    return inputs.DreamBlockCase(
        X=t(X), mask=mask.cpu().numpy(), pos=np.tile(np.arange(seq, dtype=np.int32), batch), batch=batch, seq=seq,
        hidden=H, ffn=F, heads=heads, kv_heads=kv, w_ln1=t(1 + 0.1 * _randn(g, H)), w_ln2=t(1 + 0.1 * _randn(g, H)),
        b_qkv=t(0.02 * _randn(g, nqkv)), tac=inputs.TacParams(C=H, g=128, M=t(M), d=t(d)), xf_qkv=xf(X, mask),
        xf_o=calib(H), xf_gu=calib(H), xf_down=calib(F), **{n: t(w) for n, w in W.items()})


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------
def _empty(*shape, dtype=torch.uint8):
    return torch.empty(*shape, dtype=dtype, device=DEV)


def _prepare_linear(s, dtype, order=None):
    """Weights and workspaces of one linear, laid out once."""
    L, K = s["X"].shape
    N = s["W"].shape[0]
    scheme = s["scheme"]
    W = s.pop("W")
    if order is not None:
        W = W[order].contiguous()
    s["s_w"] = _empty(N, dtype=torch.float32)
    if scheme == "w8":
        s["Wq"] = _empty(N, K)
        abi.sgat_prepare_weight(W, s["inv"], s["hb"], s["Wq"], s["s_w"], bits=8)
        s["We"] = _empty(N, 2 * K)
        abi.w8_codes_f16(s["Wq"], s["We"])
        s["Wq"] = None
        s["We"] = s["We"].view(torch.float16)
        s["ws"] = _empty(abi.sgat_linear_workspace_size(L, K, s["g"] > 0, bits=8))
    elif scheme == "dense":
        s["Wq"] = _empty(N, K // 2)
        abi.sgat_prepare_weight_dense(W, s["inv"], s["Pt"], s["Wq"], s["s_w"])
        s["We"] = _empty(N, K)
        abi.w4_unpack_e4m3(s["Wq"], s["We"])
        s["ws"] = _empty(abi.sgat_linear_dense_workspace_size(L, K))
    else:
        s["Wq"] = _empty(N, K // 2)
        abi.sgat_prepare_weight(W, s["inv"], s["hb"], s["Wq"], s["s_w"])
        if scheme == "asym":
            s["We"] = _empty(N, K + 128)
            abi.w4_zero_point_columns(s["Wq"], s["We"])
            s["ws"] = _empty(abi.sgat_linear_asym_workspace_size(L, K))
        else:
            s["We"] = _empty(N, K)
            abi.w4_unpack_e4m3(s["Wq"], s["We"])
            s["ws"] = _empty(abi.sgat_linear_workspace_size(L, K, s["g"] > 0))
    s["Mp"] = None
    if s["g"]:
        s["Mp"] = _empty(abi.tac_prepared_bytes(K, s["g"]))
        abi.tac_prepare(s["M"], s["g"], DTYPE[dtype], s["Mp"])
    s["Y"] = _empty(L, N if order is None else N // 2, dtype=DTYPE[dtype])
    return s


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "linear":
        s = _prepare_linear(_linear_inputs(g, case["L"], case["K"], case["N"], case["dtype"], case["scheme"],
                                           case["tac"], case["bias"]), case["dtype"])
    elif kind == "attn_step":
        qkv = _linear_inputs(g, case["L"], 4096, 12288, "f16")
        o = _linear_inputs(g, case["L"], 4096, 4096, "f16", tac=128)
        step = AttentionProjections(_np_linear(qkv, "f16"), _np_linear(o, "f16"), grouped=True)
        step.step()
        step.capture()
        s = dict(step=step)
    elif kind == "mlp":
        gu, down = _mlp_inputs(case, g)
        s = dict(gu=_prepare_linear(gu, case["dtype"], abi.swiglu_row_order(case["F"], DEV)),
                 down=_prepare_linear(down, case["dtype"]))
    elif kind == "attention":
        qkv, M, d = _attention_inputs(case, g)
        L, H, Hkv = case["L"], case["H"], case["Hkv"]
        Mp = _empty(abi.tac_prepared_bytes(128 * H, 128))
        abi.tac_prepare(M, 128, torch.float16, Mp)
        s = dict(qkv=qkv, H=H, Hkv=Hkv, M=M, d=d, Mp=Mp, Z=_empty(L, 128 * H, dtype=qkv.dtype),
                 ws=_empty(abi.attention_pv_tac_workspace_size(L, Hkv)))
    elif kind == "tac":
        Z = _acts(g, case["L"], case["C"], case["dtype"])
        M, d = _tac(g, case["C"], case["g"])
        Mp = None
        if case["prepared"]:
            Mp = _empty(abi.tac_prepared_bytes(case["C"], case["g"]))
            abi.tac_prepare(M, case["g"], DTYPE[case["dtype"]], Mp)
        s = dict(Z=Z, M=M, d=d, g=case["g"], Mp=Mp, out=_empty(case["L"], case["C"], dtype=DTYPE[case["out"]]))
    elif kind == "weights":
        N, K = case["N"], case["K"]
        s = dict(W=_weight(g, N, K, case["dtype"]), inv=(0.5 * _randn(g, K)).exp(), hb=inputs.hadamard_block(K),
                 Wq=_empty(N, K // 2), s_w=_empty(N, dtype=torch.float32), We=_empty(N, K))
    elif kind == "stack":
        st = DenoiseStack(StackConfig(seq=case["seq"], layers=case["layers"], seed=int(seed)))
        st.calibrate()
        graph, tok, mask, out = st.capture()
        st.set_state(case["step"], tok, mask)
        s = dict(st=st, graph=graph, tok=tok, mask=mask, out=out)     # the graph reads tok and mask
    else:
        blk = DreamBlock(_dream_case(case, g))
        blk.forward()
        blk.capture()
        s = dict(blk=blk)
    s["kind"] = kind
    return s


def _run_linear(s, X=None, swiglu=False):
    X = s["X"] if X is None else X
    d_sh, d_m, d_u = s["gate"]
    if s["scheme"] == "dense":
        abi.sgat_linear_dense(X, s["mask"], s["a_m"], s["a_u"], s["Pt"], d_sh, d_m, d_u, s["Wq"], s["s_w"], s["Y"],
                              s["ws"], bias=s["bias"], We=s["We"])
    elif s["scheme"] == "asym":
        abi.sgat_linear_asym(X, s["mask"], s["a_m"], s["a_u"], s["hb"], d_sh, d_m, d_u, s["We"], s["s_w"], s["Y"],
                             s["ws"], bias=s["bias"])
    elif swiglu:
        abi.sgat_linear_swiglu(X, s["mask"], s["a_m"], s["a_u"], s["hb"], d_sh, d_m, d_u, s["Wq"], s["s_w"], s["Y"],
                               s["ws"], We=s["We"])
    else:
        abi.sgat_linear(X, s["mask"], s["a_m"], s["a_u"], s["hb"], d_sh, d_m, d_u, s["Wq"], s["s_w"], s["Y"],
                        s["ws"], bias=s["bias"], tac_M=s["M"], tac_d=s["d"], tac_g=s["g"],
                        bits=8 if s["scheme"] == "w8" else 4, We=s["We"], tac_Mp=s["Mp"])
    return s["Y"]


def run(state):
    s = state
    kind = s["kind"]
    if kind == "linear":
        return _run_linear(s)
    if kind == "attn_step":
        s["step"].replay()
        return s["step"].Y_qkv, s["step"].Y_o
    if kind == "mlp":
        h = _run_linear(s["gu"], swiglu=True)
        return h, _run_linear(s["down"], X=h)
    if kind == "attention":
        q, c, k = s["qkv"], 128 * s["H"], 128 * s["Hkv"]
        abi.attention_pv_tac(q[:, :c], q[:, c:c + k], q[:, c + k:], s["H"], s["Mp"], s["d"], s["Z"], workspace=s["ws"],
                             Hkv=s["Hkv"])
        return s["Z"]
    if kind == "tac":
        abi.tac_apply(s["Z"], s["M"], s["d"], s["g"], s["out"], Mp=s["Mp"])
        return s["out"]
    if kind == "weights":
        abi.sgat_prepare_weight(s["W"], s["inv"], s["hb"], s["Wq"], s["s_w"])
        abi.w4_unpack_e4m3(s["Wq"], s["We"])
        return s["Wq"], s["We"], s["s_w"]
    if kind == "stack":
        s["graph"].replay()
        return s["out"]
    s["blk"].replay()
    return s["blk"].buf["out"]


# ---------------------------------------------------------------------------
# Necessary work
# ---------------------------------------------------------------------------
def _linear_work(L, K, N, scheme="w4", tac=0, extra=0):
    w = N * K if scheme == "w8" else N * K // 2
    b = 2 * L * K + L + w + 4 * N + 8 * K + 2 * L * N + 4 * K * tac + extra
    f = 2.0 * L * N * K + 2.0 * L * K * tac
    if scheme == "dense":
        b += 2 * K * K
        f += 2.0 * L * K * K
    return b, f


def _attention_work(L, H, Hkv):
    return 2 * 128 * L * (2 * H + 2 * Hkv) + 4 * 128 * 128 * H, 4.0 * L * L * 128 * H + 2.0 * L * 128 * 128 * H


def work(case):
    kind = case["kind"]
    if kind == "linear":
        b, f = _linear_work(case["L"], case["K"], case["N"], case["scheme"], case["tac"])
    elif kind == "attn_step":
        b, f = map(sum, zip(_linear_work(case["L"], 4096, 12288), _linear_work(case["L"], 4096, 4096, tac=128)))
    elif kind == "mlp":
        L, H, F = case["L"], case["H"], case["F"]
        b = 2 * L * H + L + 3 * H * F // 2 + 4 * (2 * F + H) + 2 * L * F + 2 * L * H
        f = 6.0 * L * H * F
    elif kind == "attention":
        b, f = _attention_work(case["L"], case["H"], case["Hkv"])
    elif kind == "tac":
        o = 4 if case["out"] == "f32" else 2
        b = (2 + o) * case["L"] * case["C"] + 4 * case["C"] * (case["g"] + 1)
        f = 2.0 * case["L"] * case["C"] * case["g"]
    elif kind == "weights":
        N, K = case["N"], case["K"]
        b = 2 * N * K + N * K // 2 + N * K + 4 * N + 4 * K
        f = float(N) * K * (math.log2(inputs.hadamard_block(K)) + 3)
    elif kind == "stack":
        L, H, F, n = case["seq"], 4096, 12288, case["layers"]
        b = n * ((4 * H * H + 3 * H * F) // 2 + 4 * 128 * 128 * 32) + 4 * L * H
        f = n * (2.0 * L * (4 * H * H + 3 * H * F) + _attention_work(L, 32, 32)[1])
    else:
        L, S, H, F = case["batch"] * case["seq"], case["seq"], 3584, 18944
        w = 4608 * H + H * H + 3 * H * F
        b = w // 2 + 4 * L * H + 4 * 128 * 128 * 28
        f = 2.0 * L * w + case["batch"] * _attention_work(S, 28, 4)[1]
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times the distance between the path and its float64 form
    (largest of the seeds and drawn sizes looked at): the output's rounding,
    and codes that fall the other way where a value lies next to a rounding
    boundary of the 4-bit quantiser."""
    kind = case["kind"]
    r = {"f16": 0.0015, "bf16": 0.008}.get(case.get("dtype", "f16"))       # seen: 0.00033, 0.0017
    if kind == "linear":
        if case["scheme"] == "dense":          # the transform itself is stored in fp16: seen 0.006
            return {"rel": 0.025}
        if case["scheme"] == "asym":           # seen 0.004
            return {"rel": 0.015}
        return {"rel": r + (0.012 if case["tac"] else 0.0)}                 # TAC output rounded: seen 0.0026
    if kind == "attn_step":
        return {"rel": 0.012}
    if kind == "tac":
        return {"rel": r}                      # seen 0.00021
    if kind == "weights":                      # the codes are whole numbers and stay; s_w seen 5e-8
        return {"rel": 1e-6}
    # seen: mlp 0.011 (two quantised linears in a row), attention 0.009; a
    # difference in the last bit of one layer's output grows through every
    # quantiser behind it, so the models' outputs hold only where their
    # layers stay bit for bit the same or nearly so
    return {"rel": 0.03}


# ---------------------------------------------------------------------------
# The same computations in float64
# ---------------------------------------------------------------------------
def _hadamard(v, hb):
    shape = v.shape
    h = 1
    while h < hb:
        v = v.reshape(-1, hb // (2 * h), 2, h)
        v = torch.stack([v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]], 2)
        h *= 2
    return v.reshape(shape)


def _tac64(z, M, d):
    B, G, _ = M.shape
    return (torch.einsum("lbj,brj->lbr", z.double().reshape(-1, B, G), M.double()) + d.double()).reshape(z.shape)


def _codes(v, qmax):
    a = v.abs().amax(1, keepdim=True)
    return torch.round(v * torch.where(a > 0, qmax / a, 0.0)), a / qmax


def _transform(s, X):
    K = X.shape[1]
    a = torch.where(s["mask"][:, None] == 1, s["a_m"][None], s["a_u"][None]).double()
    v = X.double() * a
    if s["scheme"] == "dense":            # the scaled rows and the transform are stored as fp16
        v = (v.half().double() @ s["Pt"].double().t()).half().double()
    else:
        v = _hadamard(v, s["hb"])
    d_sh, d_m, _ = s["gate"]
    j = torch.arange(K, device=DEV)[None]
    m = s["mask"][:, None] == 1
    return torch.where((j < d_sh) | torch.where(m, j < d_sh + d_m, j >= d_sh + d_m), v, 0.0)


def _weight_codes(s, qmax):
    w = s["W"].double() * s["inv"].double()
    if s["scheme"] == "dense":
        return _codes((w.half().double() @ s["Pt"].double().t()).half().double(), qmax)
    return _codes(_hadamard(w, s["hb"]) / s["hb"], qmax)


def _linear64(s, X=None):
    """[L][N] in float64. Sums of 4-bit codes stay below 2^24, so their
    products run in float32 and are exact."""
    X = s["X"] if X is None else X
    if s["g"]:
        X = _tac64(X, s["M"], s["d"]).to(X.dtype)
    qmax = 127.0 if s["scheme"] == "w8" else 7.0
    v = _transform(s, X)
    qw, sw = _weight_codes(s, qmax)
    if s["scheme"] == "asym":
        lo, hi = v.amin(1, keepdim=True).clamp_max(0), v.amax(1, keepdim=True).clamp_min(0)
        sa = (hi - lo) / 15
        z = torch.round(-lo / sa)
        qa = (torch.round(v / sa) + z).clamp(0, 15) - z
    else:
        qa, sa = _codes(v, qmax)
    if s["scheme"] == "w8":
        acc = qa @ qw.t()
    else:
        tf32 = torch.backends.cuda.matmul.allow_tf32
        torch.backends.cuda.matmul.allow_tf32 = False
        acc = (qa.float() @ qw.float().t()).double()
        torch.backends.cuda.matmul.allow_tf32 = tf32
    y = acc * sa * sw.t()
    return y if s["bias"] is None else y + s["bias"].double()


def _attention64(q, k, v, H, Hkv, M, d):
    L = q.shape[0]
    vq, t = _codes(v.double().t(), 7.0)                        # per channel
    out = []
    for h in range(H):
        hk = h // (H // Hkv)
        c, ck = slice(128 * h, 128 * h + 128), slice(128 * hk, 128 * hk + 128)
        sc = q[:, c].double() @ k[:, ck].double().t() / math.sqrt(128.0)
        e = torch.exp(sc - sc.amax(1, keepdim=True))
        z = (torch.round(255 * e) @ vq[ck].t()) / (255 * e.sum(1, keepdim=True)) * t[ck].t()
        out.append(z @ M[h].double().t() + d[h].double())
    return torch.cat(out, 1)


def _silu(x):
    return x * torch.sigmoid(x)


def exact(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "linear":
        return _linear64(_linear_inputs(g, case["L"], case["K"], case["N"], case["dtype"], case["scheme"], case["tac"],
                                        case["bias"]))
    if kind == "attn_step":
        qkv = _linear_inputs(g, case["L"], 4096, 12288, "f16")
        o = _linear_inputs(g, case["L"], 4096, 4096, "f16", tac=128)
        return _linear64(qkv), _linear64(o)
    if kind == "mlp":
        gu, down = _mlp_inputs(case, g)
        y = _linear64(gu)
        h = _silu(y[:, : case["F"]]) * y[:, case["F"]:]
        return h, _linear64(down, X=h.to(DTYPE[case["dtype"]]))
    if kind == "attention":
        qkv, M, d = _attention_inputs(case, g)
        c, k = 128 * case["H"], 128 * case["Hkv"]
        return _attention64(qkv[:, :c], qkv[:, c:c + k], qkv[:, c + k:], case["H"], case["Hkv"], M, d)
    if kind == "tac":
        Z = _acts(g, case["L"], case["C"], case["dtype"])
        return _tac64(Z, *_tac(g, case["C"], case["g"]))
    if kind == "weights":
        N, K = case["N"], case["K"]
        W = _weight(g, N, K, case["dtype"])
        _, s_w = _codes(_hadamard(W.double() * (0.5 * _randn(g, K)).exp().double(), inputs.hadamard_block(K))
                        / inputs.hadamard_block(K), 7.0)
        return None, None, s_w.reshape(-1)
    # The stack calibrates itself with this library's own kernels, and in both
    # models a value next to a rounding boundary decides codes that the later
    # quantisers amplify (a float64 form of the block ends 0.18 away although
    # each of its layers is within 0.011): no independent value.
    return None
