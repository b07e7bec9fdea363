"""The work this library is used for, as cases whose speed is watched.

Everything goes through the public entry points (``paper_2603_05168_b200.binding``).  Four kinds:

  infer   forward passes of the BitLinears of one or several layers on packed weights: decoding a few
          tokens, chunks and prefills; int8-held, 2-bit-packed, dense-ternary and 6:8 weights
  pack    latent weights -> packed ternary weights: the re-pack of a dynamic-mask training step (one
          batched call, the previous step's scales as hints, flip counts), or loading (one call per matrix)
  step68  re-pack and forward with the 6:8 pattern, which has no batched pack call
  train   one training step of a layer: re-pack, forward, backward (both gradients)

Sizes are those of the 2B- and 7B-shaped layers in ``inputs.py``; drawn cases move around them.
"""
from __future__ import annotations

import math

import torch

from paper_2603_05168_b200 import binding as b
from paper_2603_05168_b200 import inputs

BF16, F32 = torch.bfloat16, torch.float32


# -- which linears a case runs: (name, K = d_in, N = d_out) ----------------------------------------
def _linears(case):
    hidden, ffn, qkv = case["hidden"], case["ffn"], case["qkv"]
    if case["linears"] == "one":
        return [("o", hidden, hidden)]
    mlp = [("gate_up", hidden, ffn), ("down", ffn, hidden)]
    if case["linears"] == "mlp":
        return mlp
    if case["linears"] == "layer":
        return [("qkv", hidden, qkv), ("o", hidden, hidden)] + mlp
    # "separate": every projection is its own tensor (as LAYER_2B)
    kv = (qkv - hidden) // 2
    return [("q", hidden, hidden), ("k", hidden, kv), ("v", hidden, kv), ("o", hidden, hidden),
            ("gate", hidden, ffn), ("up", hidden, ffn), ("down", ffn, hidden)]


def _2b(**more):
    """The layer of inputs.SHAPES_2B / LAYER_2B."""
    shapes = {name: (K, N) for name, K, N in inputs.SHAPES_2B}
    return dict(hidden=shapes["o"][0], ffn=shapes["gate_up"][1], qkv=shapes["qkv"][1], heavy=False, **more)


def _7b(**more):
    """The MLP of inputs.SHAPES_7B, with the heavier-tailed weights and activations it is benchmarked on."""
    shapes = {name: (K, N) for name, K, N in inputs.SHAPES_7B}
    hidden, ffn = shapes["gate_up_7b"]
    return dict(hidden=hidden, ffn=ffn, qkv=3 * hidden, heavy=True, **more)


def _infer(T, **over):
    case = dict(kind="infer", T=T, layers=1, linears="layer", weights="sparse", norm=False, bias=False, out="bf16",
                fused=False, graph=False)
    case.update(over)
    return case


def listed():
    return [
        # the smallest call: one projection for one token, quantiser and GEMM in one entry point
        dict(_infer(1, linears="one", fused=True), **_2b(), name="one_linear_1tok"),
        # decoding one sequence, the step captured once as serving loops do; the weights of four layers
        # (more than the L2 holds) stream from memory
        dict(_infer(1, layers=4, norm=True, graph=True), **_2b(), name="decode_1tok_2b_graph"),
        # decoding a batch of 16 sequences with direct calls, wide matrices
        dict(_infer(16, layers=2, linears="mlp", norm=True), **_7b(), name="decode_16tok_7b"),
        # decoding with the weights kept at two bits each (memory capacity)
        dict(_infer(4, layers=2, linears="mlp", weights="packed"), **_7b(), name="decode_4tok_7b_packed"),
        # a prompt chunk or a large decode batch, ragged; fp32 outputs with bias
        dict(_infer(201, bias=True, out="f32"), **_2b(), name="chunk_201tok_2b_f32"),
        # a short ragged prompt through the dense-ternary layer
        dict(_infer(777, weights="dense"), **_2b(), name="prefill_777tok_2b_dense"),
        # an ordinary prefill
        dict(_infer(4096, norm=True), **_2b(), name="prefill_4096tok_2b"),
        # the largest prefill
        dict(_infer(8192, linears="mlp"), **_7b(), name="prefill_8192tok_7b"),
        # packing weights at load time: one call per matrix, bf16 masters, nothing known about them
        dict(kind="pack", layers=1, linears="layer", masters="bf16", batched=False, dense_q=False, **_2b(),
             name="load_pack_bf16_2b"),
        # the dynamic-mask re-pack of two layers (seven tensors each) in a training step
        dict(kind="pack", layers=2, linears="separate", masters="f32", batched=True, dense_q=False, **_2b(),
             name="repack_2layers_2b"),
        # re-pack and forward with the 6:8 pattern
        dict(kind="step68", T=2048, linears="layer", masters="f32", **_2b(), name="step68_2048tok_2b"),
        # one training step of a layer
        dict(kind="train", T=4096, linears="layer", masters="f32", **_2b(), name="train_4096tok_2b"),
    ]


def draw(rng):
    # none larger than the training step and the largest prefill above
    while True:
        case = _draw_any(rng)
        cost = work(case)
        if cost["bytes"] <= 0.95e9 and cost["flops"] <= (1.06e12 if case["kind"] == "train" else 0.73e12):
            return case


def _draw_any(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def m128(lo, hi):
        return 128 * rng.randint(lo // 128, hi // 128)

    kind = rng.choice(["infer"] * 8 + ["pack", "pack", "step68", "train"])
    hidden = m128(1024, 4096)
    size = dict(hidden=hidden, ffn=128 * max(1, int(hidden * rng.uniform(2.0, 3.0)) // 128),
                qkv=hidden + 256 * rng.randint(1, hidden // 256), heavy=rng.random() < 0.5)
    if kind == "infer":
        few = rng.random() < 0.5
        T = log_int(1, 64) if few else log_int(65, 8192)
        case = _infer(T, norm=rng.random() < 0.5, bias=rng.random() < 0.3, out=rng.choice(["bf16", "bf16", "f32"]))
        if few:
            case.update(linears=rng.choice(["layer", "mlp"]), layers=rng.randint(1, 3), graph=rng.random() < 0.4,
                        weights=rng.choice(["sparse"] * 4 + ["packed", "dense"]))
            if T <= 32 and case["weights"] == "sparse" and rng.random() < 0.25:
                case.update(fused=True, norm=False)
        else:
            case.update(linears=rng.choice(["layer", "mlp"]),
                        weights=rng.choice(["sparse", "sparse", "sparse", "dense"]))
        return dict(case, **size)
    masters = rng.choice(["f32", "bf16"])
    if kind == "pack":
        linears = rng.choice(["layer", "separate"])
        return dict(kind="pack", layers=rng.randint(1, 2), linears=linears, masters=masters, batched=rng.random() < 0.6,
                    dense_q=linears == "layer" and rng.random() < 0.3, **size)
    size["hidden"] = hidden = 256 * rng.randint(4, 10)                # 6:8 works on multiples of 256 columns
    size["ffn"] = 256 * max(1, int(hidden * rng.uniform(2.0, 2.7)) // 256)
    size["qkv"] = hidden + 256 * rng.randint(1, hidden // 512)
    return dict(kind=kind, T=log_int(256, 4096), linears="layer", masters=masters, **size)


# -- inputs ----------------------------------------------------------------------------------------
def _latent(gen, N, K, heavy):
    """Latent weights: N(0, 0.02^2), or N(0, 0.015^2) with 5 % of the entries ten times larger."""
    W = torch.randn((N, K), generator=gen, device="cuda", dtype=F32)
    if not heavy:
        return W.mul_(0.02)
    return W.mul_(0.015).mul_(1.0 + 9.0 * (torch.rand((N, K), generator=gen, device="cuda") < 0.05))


def _acts(gen, T, K, heavy):
    x = torch.randn((T, K), generator=gen, device="cuda", dtype=F32)
    if heavy:                                                          # per-token LogNormal(0, 0.5) scale
        x.mul_(torch.exp(0.5 * torch.randn((T, 1), generator=gen, device="cuda")))
    return x.to(BF16)


def _pack_now(W, **kw):
    bufs = b.alloc_packed(*W.shape, **kw)
    pattern = {k: v for k, v in kw.items() if k in ("n_keep", "m_group")}
    b.sbn_quantize_mask_pack(W, bufs["vals"], bufs["meta"], bufs["w_scale"], bufs["ws"], dense_q=bufs.get("dense_q"), **pattern)
    return bufs


def _prepare_infer(case, gen):
    T, mode, heavy = case["T"], case["weights"], case["heavy"]
    sources = {}                                                       # activations by linear; layers take them in turn
    linears = []
    for _ in range(case["layers"]):
        for name, K, N in _linears(case):
            if name not in sources:
                sources[name] = dict(
                    x=_acts(gen, T, K, heavy), xq=b.alloc_xq(T, K),
                    a_scale=torch.empty(T, dtype=F32, device="cuda"),
                    gain=0.5 + torch.rand(K, generator=gen, device="cuda") if case["norm"] and name in ("qkv", "gate_up") else None)
            W = _latent(gen, N, K, heavy)
            packed = _pack_now(W, with_dense=mode == "dense")
            lin = dict(sources[name], N=N, K=K, vals=packed["vals"], meta=packed["meta"], w_scale=packed["w_scale"],
                       bias=torch.randn(N, generator=gen, device="cuda") if case["bias"] else None,
                       y=torch.empty((T, N), dtype=BF16 if case["out"] == "bf16" else F32, device="cuda"))
            if mode == "packed":
                lin["vals2"] = b.alloc_vals2(N, K)
                b.sbn_pack_vals2(lin.pop("vals"), lin["vals2"])
            elif mode == "dense":
                lin["dense_q"] = packed["dense_q"]
                del lin["vals"], lin["meta"]
            if mode != "packed":
                lin["ws"] = b.alloc_gemm_ws(b.OP_BITLINEAR if mode == "dense" else b.OP_SPARSE_BITLINEAR, T, N, K)
            linears.append(lin)
    state = dict(case=case, linears=linears, out=[lin["y"] for lin in linears], graph=None)
    if case["graph"]:
        _run_infer(state)
        torch.cuda.synchronize()
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            _run_infer(state)
    return state


def _prepare_pack(case, gen):
    masters = F32 if case["masters"] == "f32" else BF16
    mats = []
    for _ in range(case["layers"]):
        for _, K, N in _linears(case):
            W = _latent(gen, N, K, case["heavy"])
            mat = dict(b.alloc_packed(N, K, with_dense=case["dense_q"]))
            if case["batched"]:
                # a training step: the masks and scales of the step before are at hand, and the weights moved a little
                before = _pack_now(W)
                mat.update(prev_meta=before["meta"], gamma_hint=before["w_scale"],
                           flip_bits=torch.zeros(1, dtype=torch.int64, device="cuda"))
                W = W.add_(torch.randn((N, K), generator=gen, device="cuda"), alpha=1e-4)
            mat["W"] = W.to(masters)
            mats.append(mat)
    state = dict(case=case, mats=mats)
    if case["batched"]:
        state["jobs"] = b.make_pack_jobs(mats)
        state["ws"] = torch.empty(b.sbn_batch_workspace_bytes(len(mats)), dtype=torch.uint8, device="cuda")
    else:
        state["ws"] = mats[0]["ws"]                                    # one scratch for all matrices, as a loader has
    keys = [k for k in ("vals", "meta", "w_scale", "dense_q", "flip_bits") if k in mats[0]]
    state["out"] = [{k: m[k] for k in keys} for m in mats]
    return state


def _prepare_step68(case, gen):
    masters, T, linears = (F32 if case["masters"] == "f32" else BF16), case["T"], []
    for _, K, N in _linears(case):
        lin = dict(b.alloc_packed(N, K, n_keep=6, m_group=8), N=N, K=K, W=_latent(gen, N, K, case["heavy"]).to(masters),
                   x=_acts(gen, T, K, case["heavy"]), xq=b.alloc_xq(T, b.sbn_expanded_k(K, 6, 8)),
                   a_scale=torch.empty(T, dtype=F32, device="cuda"), y=torch.empty((T, N), dtype=BF16, device="cuda"))
        lin["gemm_ws"] = b.alloc_gemm_ws(b.OP_SPARSE_BITLINEAR, T, N, b.sbn_expanded_k(K, 6, 8))
        linears.append(lin)
    return dict(case=case, linears=linears, out=[{k: m[k] for k in ("vals", "meta", "w_scale", "y")} for m in linears])


def _prepare_train(case, gen):
    pack = _prepare_pack(dict(case, layers=1, batched=True, dense_q=False), gen)
    T, linears = case["T"], []
    for (_, K, N), mat in zip(_linears(case), pack["mats"]):
        linears.append(dict(
            mat, N=N, K=K, x=_acts(gen, T, K, case["heavy"]), xq=b.alloc_xq(T, K),
            a_scale=torch.empty(T, dtype=F32, device="cuda"), y=torch.empty((T, N), dtype=BF16, device="cuda"),
            dY=torch.randn((T, N), generator=gen, device="cuda").mul_(1e-3).to(BF16),
            dX=torch.empty((T, K), dtype=BF16, device="cuda"), dW=torch.empty((N, K), dtype=F32, device="cuda"),
            gemm_ws=b.alloc_gemm_ws(b.OP_SPARSE_BITLINEAR, T, N, K)))
    need = max(b.sbn_workspace_bytes(b.OP_BACKWARD, T, m["N"], m["K"]) for m in linears)
    return dict(case=case, linears=linears, jobs=pack["jobs"], ws=pack["ws"],
                back_ws=torch.empty(need, dtype=torch.uint8, device="cuda"),
                out=[{k: m[k] for k in ("vals", "meta", "w_scale", "flip_bits", "y", "dX", "dW")} for m in linears])


_PREPARE = dict(infer=_prepare_infer, pack=_prepare_pack, step68=_prepare_step68, train=_prepare_train)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return _PREPARE[case["kind"]](case, gen)


# -- one pass --------------------------------------------------------------------------------------
def _run_infer(state):
    case = state["case"]
    mode, fused = case["weights"], case["fused"]
    for lin in state["linears"]:
        if fused:
            b.sbn_quant_act_sparse_bitlinear(lin["x"], lin["vals"], lin["meta"], lin["w_scale"], lin["y"], bias=lin["bias"])
            continue
        if lin["gain"] is not None:
            b.sbn_norm_quant_act(lin["x"], lin["xq"], lin["a_scale"], gain=lin["gain"])
        else:
            b.sbn_quant_act(lin["x"], lin["xq"], lin["a_scale"])
        if mode == "sparse":
            b.sbn_sparse_bitlinear(lin["xq"], lin["a_scale"], lin["vals"], lin["meta"], lin["w_scale"], lin["y"], bias=lin["bias"], ws=lin["ws"])
        elif mode == "packed":
            b.sbn_sparse_bitlinear_packed(lin["xq"], lin["a_scale"], lin["vals2"], lin["meta"], lin["w_scale"], lin["y"], bias=lin["bias"])
        else:
            b.sbn_bitlinear(lin["xq"], lin["a_scale"], lin["dense_q"], lin["w_scale"], lin["y"], bias=lin["bias"], ws=lin["ws"])


def _run_pack(state):
    if "jobs" in state:
        b.sbn_quantize_mask_pack_batched(state["jobs"], state["ws"])
    else:
        for m in state["mats"]:
            b.sbn_quantize_mask_pack(m["W"], m["vals"], m["meta"], m["w_scale"], state["ws"], dense_q=m.get("dense_q"))


def _run_step68(state):
    for m in state["linears"]:
        b.sbn_quantize_mask_pack(m["W"], m["vals"], m["meta"], m["w_scale"], m["ws"], n_keep=6, m_group=8)
        b.sbn_quant_act_expand68(m["x"], m["xq"], m["a_scale"])
        b.sbn_sparse_bitlinear(m["xq"], m["a_scale"], m["vals"], m["meta"], m["w_scale"], m["y"], ws=m["gemm_ws"])


def _run_train(state):
    b.sbn_quantize_mask_pack_batched(state["jobs"], state["ws"])
    for m in state["linears"]:
        b.sbn_quant_act(m["x"], m["xq"], m["a_scale"])
        b.sbn_sparse_bitlinear(m["xq"], m["a_scale"], m["vals"], m["meta"], m["w_scale"], m["y"], ws=m["gemm_ws"])
    for m in reversed(state["linears"]):
        b.sbn_bitlinear_backward(m["dY"], m["xq"], m["a_scale"], m["vals"], m["meta"], m["w_scale"], m["N"], m["K"],
                                 dX=m["dX"], dW=m["dW"], ws=state["back_ws"])


_RUN = dict(infer=_run_infer, pack=_run_pack, step68=_run_step68, train=_run_train)


def run(state):
    if state.get("graph") is not None:
        state["graph"].replay()
    else:
        _RUN[state["case"]["kind"]](state)
    return state["out"]


# -- what a pass cannot do without -----------------------------------------------------------------
def work(case):
    kind, T = case["kind"], case.get("T", 0)
    nbytes = flops = 0.0
    for _, K, N in _linears(case):
        if kind == "infer":
            per_weight = dict(sparse=0.625, packed=0.25, dense=1.0)[case["weights"]]
            nbytes += per_weight * N * K + 2.0 * T * K + (2.0 if case["out"] == "bf16" else 4.0) * T * N
            flops += (2.0 if case["weights"] == "dense" else 1.0) * T * N * K     # only kept weights are multiplied
            continue
        masters = 4.0 if case["masters"] == "f32" else 2.0
        kept = 0.9375 if kind == "step68" else 0.625                              # bytes per weight of the packed form
        nbytes += (masters + kept) * N * K
        if kind == "pack":
            nbytes += ((1.0 if case["dense_q"] else 0.0) + (0.125 if case["batched"] else 0.0)) * N * K
        elif kind == "step68":
            nbytes += 2.0 * T * (K + N)
            flops += 1.5 * T * N * K
        else:
            nbytes += 0.125 * N * K + 4.0 * T * (K + N) + 4.0 * N * K             # x, dX, y, dY in bf16; dW in fp32
            flops += (1.0 + 2.0 + 2.0) * T * N * K
    layers = case.get("layers", 1)
    return {"bytes": nbytes * layers, "flops": flops * layers}


def tolerance(case):
    """Integer sums are exact and packed bytes and masks unique, so outputs differ by the roundings of fp32
    scales only: the scale one unit off (its fp64 sum in another order) or the factors of a dequantisation in
    another order measured rel 1.3e-7 / max 3.3e-7 in fp32 outputs, and rel 4e-5 / one unit in the last place
    in bf16 ones.  Gradients are fp32 sums of exact products; against sums in fp64, dX (bf16) measured rel
    2e-5 / one unit, dW (fp32) rel 4e-6 / max 2e-5.  About four times the larger is stated."""
    if case["kind"] == "infer" and case["out"] == "f32":
        return {"rel": 5e-7, "max": 1.3e-6}
    if case["kind"] == "pack":
        return {"rel": 5e-7, "max": 5e-7}
    return {"rel": 1.5e-4, "max": 8e-3}
