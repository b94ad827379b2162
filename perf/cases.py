"""The calls that this library's performance is measured on, as a user's program makes them (see `binding` and `ep`).

Three ways of using the library are covered, each over its whole range of sizes:

* ``layer``  one MoE layer of a serving model: `moe_layer` (bf16 experts) or `moe_layer_fp8` (E4M3 experts, quantised once
  when the model is loaded), from the single token of a decode step to the tens of thousands of a prefill batch;
* ``train``  one training step of the layer: `moe_layer` with its routing kept, `moe_layer_backward`, `moe_gate_backward`;
* ``ep``     what one rank of an expert-parallel layer computes (`ep.EpRank`): its send phase, its experts on the rows it
  received, and the final reduction.  The exchange over the links is left out: rows come back as they went.

Shapes are those of `synth.ALL_CONFIGS` (expert widths, expert counts, top-k, groups, router bias) with batch sizes of use.
"""
from __future__ import annotations

import math

import torch

from paper_2605_05607_b200 import binding as B
from paper_2605_05607_b200 import ep
from paper_2605_05607_b200 import synth

SOFTMAX, SIGMOID = synth.SCORE_SOFTMAX, synth.SCORE_SIGMOID


def _case(name, use, T, d, f, E, k, G, score=SOFTMAX, bias="none", dtype="bf16"):
    c = {"use": use, "T": T, "d": d, "f": f, "E": E, "k": k, "G": G, "score": score, "bias": bias, "dtype": dtype}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest layer of the configurations: launches and latency count, not bytes
        _case("tiny layer", "layer", 256, 512, 1024, 8, 2, 4),
        # one token of one sequence: two wide Mixtral-shaped experts are read for it
        _case("decode 1 token", "layer", 1, 4096, 14336, 8, 2, 8),
        # a decode batch: nearly all of 128 Qwen3-shaped experts are read for a handful of rows each
        _case("decode 64 tokens", "layer", 64, 4096, 1536, 128, 8, 8),
        # a larger decode batch on DeepSeek-V3-shaped experts stored in 8 bits
        _case("decode 128 tokens fp8", "layer", 128, 7168, 2048, 256, 8, 8, SIGMOID, dtype="fp8"),
        # a short prompt on GPT-OSS-shaped experts with popular and unpopular ones; sizes that no tile divides
        _case("prefill 1777 skewed", "layer", 1777, 2880, 2880, 128, 4, 8, bias="zipf"),
        # a prefill batch on few wide experts
        _case("prefill 4096 wide", "layer", 4096, 4096, 14336, 8, 2, 8),
        # a prefill batch on many narrow experts in 8 bits, tokens favouring one group
        _case("prefill 16384 fp8", "layer", 16384, 4096, 1536, 128, 8, 8, bias="locality", dtype="fp8"),
        # the largest: a full prefill batch on 256 DeepSeek-V3-shaped experts
        _case("prefill 32768", "layer", 32768, 7168, 2048, 256, 8, 8, SIGMOID),
        # training of the paper's Small layer at top-8
        _case("train small layer", "train", 8192, 2048, 512, 64, 8, 32, SIGMOID),
        # training on skewed experts, a ragged batch
        _case("train 3001 skewed", "train", 3001, 2880, 2880, 128, 4, 8, bias="zipf"),
        # training on many experts with locality
        _case("train 8192", "train", 8192, 4096, 1536, 128, 8, 8, bias="locality"),
        # one of eight ranks of an expert-parallel layer, 16 experts of its own
        _case("ep rank", "ep", 2050, 4096, 1536, 128, 8, 8),
    ]


# largest listed case, which bounds the drawn ones
_MAX_FLOPS = 6.0 * 32768 * 8 * 7168 * 2048
_MAX_WEIGHTS = 256 * 3 * 7168 * 2048      # elements
_LOG = lambda rng, lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    while True:
        use = rng.choices(("layer", "train", "ep"), (6, 3, 1))[0]
        dtype = "fp8" if use == "layer" and rng.random() < 0.35 else "bf16"
        E = rng.choice((8, 16, 32, 64, 128, 256))
        G = rng.choice([g for g in (1, 2, 4, 8, 16, 32) if g <= E and (use != "ep" or g >= 2)])
        k = rng.choice([v for v in (1, 2, 4, 6, 8, 16) if v <= E // 2])
        d = 16 * _LOG(rng, 512 // 16, 7168 // 16)
        f = 16 * _LOG(rng, 512 // 16, 14336 // 16)
        T = _LOG(rng, 1 if use == "layer" else 256, 32768)
        factor = {"layer": 1.0, "train": 3.7, "ep": 1.0}[use]
        weights = E * 3 * d * f
        room = {"layer": 1.0, "train": 0.35, "ep": float(G)}[use] * _MAX_WEIGHTS
        rows = T * k * (2 * d + 2 * f) * (1.0 if use == "layer" else 2.5)
        if factor * 6.0 * T * k * d * f <= _MAX_FLOPS and weights <= room and rows <= 6e9:
            break
    return _case(None, use, T, d, f, E, k, G, rng.choice((SOFTMAX, SIGMOID)), rng.choice(("none", "zipf", "locality")),
                 dtype)


def _config(case):
    return synth.MoEConfig("case", T=case["T"], d=case["d"], f=case["f"], E=case["E"], k=case["k"], G=case["G"],
                           score_fn=case["score"], bias=case["bias"], zipf_s=1.1, boost=2.0)


def _normal(gen, shape, std=1.0):
    t = torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    return t if std == 1.0 else t.mul_(std)


def _quantised(w):
    E, K, N = w.shape
    q = torch.empty(E, N, K, dtype=torch.uint8, device="cuda")
    s = torch.empty(E, N, dtype=torch.float32, device="cuda")
    B.moe_quantize_weights(w, q, s)
    return q, s


def prepare(case, seed):
    cfg = _config(case).with_(seed=seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    T, d, f, E, k = cfg.T, cfg.d, cfg.f, cfg.E, cfg.k
    here = cfg.m if case["use"] == "ep" else E       # experts whose weights this GPU holds
    st = {"case": case, "x": _normal(gen, (T, d)), "bias": synth.make_bias(cfg, "cuda"),
          "w_gate": torch.randn(d, E, generator=gen, device="cuda") * 0.02}
    w1 = _normal(gen, (here, d, f), 1 / math.sqrt(d))
    w3 = _normal(gen, (here, d, f), 1 / math.sqrt(d))
    w2 = _normal(gen, (here, f, d), 1 / math.sqrt(f))
    if case["use"] == "ep":
        rank = ep.EpRank(cfg, 0, st["w_gate"], st["bias"], w1, w3, w2)
        # rows received from the ranks: as many as a balanced exchange brings, each with 1 .. kk experts of this rank
        p_miss = 1.0
        for i in range(k):
            p_miss *= (E - here - i) / (E - i) if E - here - i > 0 else 0.0
        R = max(1, round(T * cfg.G * (1 - p_miss)))
        kk = rank.kk
        score = torch.rand(R, here, generator=gen, device="cuda")
        idx = score.topk(kk, dim=1).indices.to(torch.int32)
        used = 1 + (torch.rand(R, kk - 1, generator=gen, device="cuda") < (k - 1) / (cfg.G * max(kk - 1, 1))).sum(1)
        idx[torch.arange(kk, device="cuda")[None, :] >= used[:, None]] = -1
        st.update(rank=rank, rows=_normal(gen, (R, d)), idx=idx, w=torch.rand(R, kk, generator=gen, device="cuda") / k)
        return st
    shape = B.make_shape(cfg)
    st.update(shape=shape, ws=B.alloc_workspace(shape), y=torch.empty(T, d, dtype=torch.bfloat16, device="cuda"))
    if case["dtype"] == "fp8":
        st["weights"] = _quantised(w1) + _quantised(w3) + _quantised(w2)
        return st
    st["weights"] = (w1, w3, w2)
    if case["use"] == "train":
        st.update(dy=_normal(gen, (T, d)), logits=torch.empty(T, E, device="cuda"),
                  topk_idx=torch.empty(T * k, dtype=torch.int32, device="cuda"),
                  topk_w=torch.empty(T * k, device="cuda"), layout=B.alloc_layout(shape),
                  dx=torch.empty(T, d, dtype=torch.bfloat16, device="cuda"), dw=tuple(torch.empty_like(w) for w in (w1, w3, w2)),
                  dw_gate=torch.empty(d, E, device="cuda"),
                  bws=torch.zeros(B.moe_backward_workspace_bytes(shape), dtype=torch.uint8, device="cuda"))
    return st


def run(st):
    case = st["case"]
    if case["use"] == "ep":
        rank = st["rank"]
        out = rank.send_phase(st["x"])
        partial = rank.recv_phase(st["rows"], st["idx"], st["w"])
        y = rank.finish_phase(out.rows)
        return {"y": y, "partial": partial, "topk_idx": rank.idx[: case["T"] * case["k"]],
                "topk_w": rank.w[: case["T"] * case["k"]]}
    if case["use"] == "train":
        B.moe_layer(st["shape"], st["x"], st["w_gate"], st["bias"], *st["weights"], st["y"], st["ws"], logits=st["logits"],
                    topk_idx=st["topk_idx"], topk_w=st["topk_w"], layout=st["layout"])
        B.moe_layer_backward(st["shape"], st["x"], st["dy"], st["topk_idx"], st["topk_w"], st["layout"], *st["weights"],
                             st["dx"], *st["dw"], st["bws"])
        B.moe_gate_backward(st["shape"], st["logits"], st["bias"], st["topk_idx"], st["topk_w"], st["layout"], st["w_gate"],
                            st["dx"], st["dw_gate"], st["bws"])
        return {"y": st["y"], "dx": st["dx"], "dw": st["dw"], "dw_gate": st["dw_gate"]}
    layer = B.moe_layer_fp8 if case["dtype"] == "fp8" else B.moe_layer
    layer(st["shape"], st["x"], st["w_gate"], st["bias"], *st["weights"], st["y"], st["ws"])
    return st["y"]


def _reached(case):
    """Expected number of experts that at least one token reaches (uniform routing; less when skewed)."""
    E, k, T = case["E"], case["k"], case["T"]
    if case["bias"] == "zipf":
        p = [(i + 1) ** -1.1 for i in range(E)]
        s = sum(p)
        return sum(1 - (1 - min(1.0, k * v / s)) ** T for v in p)
    return E * (1 - (1 - k / E) ** T)


def work(case):
    T, d, f, E, k, G = (case[n] for n in ("T", "d", "f", "E", "k", "G"))
    row, expert = 2 * d, 3 * d * f * (1 if case["dtype"] == "fp8" else 2)
    gate_bytes, gate_flops = 4 * d * E, 2 * T * d * E
    ffn = 6 * d * f                                    # flops of one (token, expert) pair, forward
    if case["use"] == "ep":
        copies = G * (1 - (1 - 1 / G) ** k)            # destinations of a token
        R, m = T * copies, E // G
        return {"bytes": T * row + gate_bytes + 2 * T * copies * row + T * row + 2 * R * row + m * expert,
                "flops": gate_flops + T * k * ffn}
    layer = {"bytes": 2 * T * row + gate_bytes + _reached(case) * expert, "flops": gate_flops + T * k * ffn}
    if case["use"] == "train":                         # x, dy, weights in; y, dx and the gradients out
        return {"bytes": layer["bytes"] + 2 * T * row + gate_bytes + E * expert, "flops": 3 * layer["flops"]}
    return layer


def tolerance(case):
    # Four times what the outputs differ by (2-norm) from the same path in 64 bits without intermediate rounding: y 2.9e-3
    # with bf16 experts, the gradients 2.8e-3 to 4.1e-3; with 8-bit experts 6.7e-3 from a 64-bit form that quantises h
    # itself, where a code of h can round the other way.
    tol = {"rel": 2.5e-2 if case["dtype"] == "fp8" else 1.6e-2 if case["use"] == "train" else 1.2e-2}
    if case["use"] == "ep":
        tol["differ"] = 2e-3                           # experts whose keys tie within the rounding of the logits
    return tol
