"""The calls that a serving program makes of this library, as timing cases.

A case is one pass through the public Python entry points (`paper_2511_18793_b200.binding.Engine`) on inputs of this
repository's own workload shapes (`synth.WORKLOADS`).  Operations:

  request   prefill of a batch of histories, then one decode: what a user waits for
  decode    one decode of an already prefilled batch (the step that `bench.py` quotes)
  prefill   the prompt pass of a batch, and the hidden states h_0..h_L that it leaves
  contains  validity of code tuples: Eq. 4 packing + Eq. 5 hash probe
  build     the hash set and the prefix map rebuilt from a catalogue, then a probe of the new table

Modes: 0 = draft head + hash filter alone, 1 = drafted and verified, 2 = plain beam search.  `drafts` of mode 1: "natural" =
the head's own tree (an untrained head's drafts are rejected: the mode's slow end), "tree" = the true beam sets handed
in as the draft tree (everything accepted: its fast end).

Weights: random, at the scale of a trained model's residual stream: unit embeddings, output projections divided by
sqrt(2 layers), logits of standard deviation 1/2.  Catalogue: every prefix of L - 1 codes continues to at least one item, as for the prefixes a trained model
keeps in its beam, so that every request returns `beam` items and no score is a padding value; for mode 0 43 % of the
last codes of a prefix are items, the share of valid tuples among drafted ones that the paper reports.

Outputs: the scores, and the item counts, of every request.  The codes of a bf16 decode are left out: neighbours in a beam
of 10 to 50 are a few hundredths apart, less than two correct bf16 pipelines differ by, so their order is no function
of the inputs (the sorted scores are).  The fp32 shape, where the order is one, returns its codes, and so do the
membership cases.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_2511_18793_b200 import binding, synth

DEV = "cuda"
#: No drawn case costs more flops than the largest listed one (the 7B shape's prompt chunk), nor holds more tokens.
MAX_FLOPS = 1.8e14
MAX_TUPLES = 1 << 24
MAX_ITEMS = 1 << 25


def listed():
    return [
        # the smallest engine (fp32, CUDA-core kernels): the floor of a call's launches and host work
        {"name": "tiny_decode", "op": "decode", "shape": "tiny", "mode": 1, "drafts": "natural", "batch": 4, "beam": 5, "items": 20, "ragged": False},
        # a re-ranker filters the candidates of a few requests: one small membership call
        {"name": "contains_4k", "op": "contains", "table": 1_000_000, "tuples": 4_096},
        # an offline job filters a day's candidates against the catalogue
        {"name": "contains_16m", "op": "contains", "table": 10_000_000, "tuples": MAX_TUPLES},
        # the catalogue is refreshed
        {"name": "build_10m", "op": "build", "table": 10_000_000, "tuples": 65_536},
        # the paper's latency setting: one user, beam 10, a dozen items; its own algorithm (draft head + hash filter)
        {"name": "paper_1_draft", "op": "request", "shape": "paper", "mode": 0, "drafts": "natural", "batch": 1, "beam": 10, "items": 12, "ragged": False},
        # the same user, drafted and verified by the primary model
        {"name": "paper_1_verified", "op": "request", "shape": "paper", "mode": 1, "drafts": "natural", "batch": 1, "beam": 10, "items": 12, "ragged": False},
        # a handful of users with histories of unequal length, an odd beam, plain beam search
        {"name": "paper_5_plain", "op": "request", "shape": "paper", "mode": 2, "drafts": "natural", "batch": 5, "beam": 9, "items": 29, "ragged": True},
        # a small model that serves many users at once
        {"name": "small_64_verified", "op": "decode", "shape": "small", "mode": 1, "drafts": "natural", "batch": 64, "beam": 10, "items": 50, "ragged": False},
        # an ordinary batch on a mid-size model, ragged, prompt included
        {"name": "0.5b_97_plain", "op": "request", "shape": "0.5b", "mode": 2, "drafts": "natural", "batch": 97, "beam": 20, "items": 100, "ragged": True},
        # wide beams, drafts accepted
        {"name": "1.5b_128_tree", "op": "decode", "shape": "1.5b", "mode": 1, "drafts": "tree", "batch": 128, "beam": 50, "items": 200, "ragged": False},
        # the largest decode: long histories on the 7B shape
        {"name": "7b_32_verified", "op": "decode", "shape": "7b", "mode": 1, "drafts": "natural", "batch": 32, "beam": 20, "items": 500, "ragged": False},
        # the largest prompt pass: 16 k tokens
        {"name": "7b_8_prefill", "op": "prefill", "shape": "7b", "batch": 8, "items": 500, "ragged": False},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("contains", "build", "model", "model", "model", "model", "model", "model", "model", "model"))
    if kind != "model":
        return {"op": kind, "table": _log(rng, 57_000, MAX_ITEMS), "tuples": _log(rng, 1_000, MAX_TUPLES if kind == "contains" else 65_536)}
    shape = rng.choice(("tiny", "paper", "paper", "small", "0.5b", "1.5b", "7b"))
    w = synth.WORKLOADS[shape]
    op = rng.choice(("request", "decode", "prefill"))
    case = {"op": op, "shape": shape, "batch": _log(rng, 1, max(4, w.batch)), "items": _log(rng, 3, w.n_hist), "ragged": rng.random() < 0.5}
    if op != "prefill":
        mode = rng.choice((0, 1, 1, 2)) if w.L == 3 else rng.choice((1, 1, 2))
        # (at least 8 beams: of 64 drafted tuples, mode 0, fewer than 8 are never valid; and where two prefixes tie for the last
        # place of a beam, modes 1 and 2, the choice moves one score of eight and not the result)
        case.update(mode=mode, beam=_log(rng, 8, max(20, w.beam)), drafts=rng.choice(("natural", "tree")) if mode == 1 else "natural")
    while work(case)["flops"] > MAX_FLOPS and case["batch"] > 1:
        case["batch"] = max(1, case["batch"] * 2 // 3)
    return case


# ----------------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------------

def _weights(w, gen):
    """Random weights of a shape, drawn in the storage type; see the module's text."""
    dt, d, hd = synth.torch_dtype(w), w.d_model, w.head_dim

    def mat(rows, cols, std=0.02):
        return torch.empty(rows, cols, dtype=dt, device=DEV).normal_(0.0, std, generator=gen)

    def gain(n):
        return (1.0 + 0.1 * torch.randn(n, device=DEV, generator=gen)).to(dt)

    out_std = 0.02 / math.sqrt(2.0 * w.n_layers)
    out = {"embed": mat(w.vocab, d, 1.0), "lm_head": mat(w.vocab, d, 0.5 / math.sqrt(d)), "final_norm": gain(d)}
    out.update({k: [] for k in ("attn_norm", "wq", "wk", "wv", "wo", "mlp_norm", "w_gate", "w_up", "w_down")})
    for _ in range(w.n_layers):
        out["attn_norm"].append(gain(d))
        out["wq"].append(mat(w.n_q_heads * hd, d))
        out["wk"].append(mat(w.n_kv_heads * hd, d))
        out["wv"].append(mat(w.n_kv_heads * hd, d))
        out["wo"].append(mat(d, w.n_q_heads * hd, out_std))
        out["mlp_norm"].append(gain(d))
        out["w_gate"].append(mat(w.d_ffn, d))
        out["w_up"].append(mat(w.d_ffn, d))
        out["w_down"].append(mat(d, w.d_ffn, out_std))
    out["draft_logit"] = [mat(w.T[l], d) for l in range(w.L)]
    out["draft_ws"], out["draft_we"] = mat(d, d), mat(d, d)
    out["draft_b"] = mat(1, d).reshape(d)
    return out


def _unrank(prefix, last, T):
    """int32 [n, L] tuples from the rank of the first L - 1 codes (first code most significant) and the last code."""
    cols = []
    for t in reversed(T[:-1]):
        cols.append((prefix % t).to(torch.int32))
        prefix = prefix // t
    return torch.stack(cols[::-1] + [last.to(torch.int32)], dim=1).contiguous()


def _dense_catalogue(T, gen, share):
    """Every prefix of L - 1 codes with 1, 2 or 3 last codes, or (share > 0) with about `share` of them; in random order."""
    n_prefix, t_last = math.prod(T[:-1]), T[-1]
    if share > 0:
        per = torch.full((n_prefix,), max(1, round(share * t_last)), device=DEV)
    else:
        per = torch.randint(1, 4, (n_prefix,), device=DEV, generator=gen)
    start = torch.randint(0, t_last, (n_prefix,), device=DEV, generator=gen)
    stride = torch.randint(0, t_last // 2, (n_prefix,), device=DEV, generator=gen) * 2 + 1      # odd: distinct modulo a power of two
    owner = torch.repeat_interleave(torch.arange(n_prefix, device=DEV), per)
    within = torch.arange(owner.numel(), device=DEV) - (torch.cumsum(per, 0) - per)[owner]
    last = (start[owner] + stride[owner] * within) % t_last
    return _unrank(owner, last, T)[torch.randperm(owner.numel(), device=DEV, generator=gen)].contiguous()


def _clustered_catalogue(T, gen, n):
    """n tuples whose prefixes are clustered by a power law (some tuples repeat, as in a catalogue joined from several sources)."""
    n_prefix = math.prod(T[:-1])
    rank = (n_prefix * torch.rand(n, device=DEV, generator=gen, dtype=torch.float64) ** 3).to(torch.int64).clamp_(max=n_prefix - 1)
    prefix = (rank * 2_654_435_761 + 12_345) % n_prefix                                         # popular prefixes anywhere in the space
    return _unrank(prefix, torch.randint(0, T[-1], (n,), device=DEV, generator=gen), T)


def _tuples(T, gen, catalogue, n):
    """n tuples, half of them drawn from the catalogue, half uniform over the code space, mixed."""
    member = catalogue[torch.randint(0, catalogue.shape[0], (n // 2,), device=DEV, generator=gen)]
    other = torch.stack([torch.randint(0, t, (n - n // 2,), device=DEV, generator=gen, dtype=torch.int32) for t in T], dim=1)
    return torch.cat([member, other])[torch.randperm(n, device=DEV, generator=gen)].contiguous()


def _workload(case):
    if case["op"] in ("contains", "build"):
        # the code space of four levels of 256 codes; the smallest backbone carries the table
        return synth.scaled(synth.WORKLOADS["small"], n_layers=1, d_model=64, n_q_heads=1, n_kv_heads=1, d_ffn=64, batch=1, beam=1, n_hist=1)
    return synth.scaled(synth.WORKLOADS[case["shape"]], batch=case["batch"], beam=case.get("beam", 1), n_hist=case["items"])


def prepare(case, seed):
    w, op = _workload(case), case["op"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 1_000_003 + 17)
    s = SimpleNamespace(case=case, w=w, stream=torch.cuda.Stream())     # (a stream of its own: its rounds replay as graphs)
    # a membership table has clustered prefixes; a model's, every prefix that its beams can reach
    if op in ("contains", "build"):
        catalogue = _clustered_catalogue(w.T, gen, case["table"])
    else:
        catalogue = _dense_catalogue(w.T, gen, 0.43 if case.get("mode") == 0 else 0.0)
    weights = _weights(w, gen)
    torch.cuda.synchronize()
    s.eng = binding.Engine(binding.make_config(w), weights, catalogue, w.load_factor, stream=s.stream)
    s.eng.build_hashset()
    del weights                                          # (the engine has its own copies)
    if op in ("contains", "build"):
        s.tuples = _tuples(w.T, gen, catalogue, case["tuples"])
        torch.cuda.synchronize()
        s.keys = s.eng.pack(s.tuples)
    else:
        # recent interactions: catalogue items by a power law over its order
        u = torch.rand(w.batch, w.n_hist, device=DEV, generator=gen)
        s.hist = catalogue[(catalogue.shape[0] * u ** 4).to(torch.int64).clamp_(max=catalogue.shape[0] - 1)].contiguous()
        s.n_hist = torch.full((w.batch,), w.n_hist, dtype=torch.int32, device=DEV)
        if case["ragged"]:
            s.n_hist = torch.randint(1, w.n_hist + 1, (w.batch,), dtype=torch.int32, device=DEV, generator=gen)
        torch.cuda.synchronize()
        if op == "decode" or case.get("drafts") == "tree":
            s.eng.prefill(s.hist, s.n_hist)
        if case.get("drafts") == "tree":
            beams = s.eng.decode(w.beam, mode=binding.MODE_AR, trace=True)["trace"]["beams"]
            s.tree = (beams.clone(), (beams[:, :, :, 0] >= 0).sum(dim=2).to(torch.int32).contiguous())
        if op != "prefill":
            s.out = s.eng.alloc_outputs(w.batch, w.beam)     # result buffers that the program keeps
    torch.cuda.synchronize()
    return s


def run(s):
    case, op = s.case, s.case["op"]
    with torch.cuda.stream(s.stream):
        if op == "contains":
            return s.eng.probe(s.eng.pack(s.tuples))
        if op == "build":
            unique = s.eng.build_hashset()
            return unique, s.eng.probe(s.keys)
        if op == "prefill":
            s.eng.prefill(s.hist, s.n_hist)
            return s.eng.get_hidden()
        if op == "request":
            s.eng.prefill(s.hist, s.n_hist)
        if case["drafts"] == "tree":
            out = s.eng.decode_with_draft_tree(case["beam"], s.tree[0], s.tree[1], out=s.out)
        else:
            out = s.eng.decode(case["beam"], mode=case["mode"], out=s.out)
        got = {"scores": out["scores"], "count": out["count"]}
        if s.w.dtype == "fp32":
            got["codes"] = out["codes"]
        return got


# ----------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------------------------------

def work(case):
    w, op = _workload(case), case["op"]
    if op == "contains":     # codes in, answers out, one 32-byte bucket a tuple
        return {"bytes": case["tuples"] * (4.0 * w.L + 1 + 32), "flops": 0.0}
    if op == "build":        # catalogue in, the table's slots out (load factor 0.5); then the probe
        return {"bytes": case["table"] * (4.0 * w.L + 16) + case["tuples"] * 41.0, "flops": 0.0}
    esz = 4 if w.dtype == "fp32" else 2
    hq, hkv = w.n_q_heads * w.head_dim, w.n_kv_heads * w.head_dim
    layer = (hq + 2 * hkv) * w.d_model + hq * w.d_model + 3 * w.d_ffn * w.d_model
    ctx = 1 + w.n_hist * w.L * (0.5 if case["ragged"] else 1.0)
    total = {"bytes": 0.0, "flops": 0.0}
    if op != "decode":
        tokens = w.batch * (ctx + w.L)
        total["flops"] += tokens * w.n_layers * (2.0 * layer + 2.0 * hq * (ctx + w.L))
        total["bytes"] += esz * w.n_layers * (layer + 2.0 * tokens * hkv) + 4.0 * w.batch * (w.L + 1) * w.d_model
    if op != "prefill":
        head = 2.0 * w.batch * w.beam * w.d_model * (sum(w.T) + (w.L - 1) * w.d_model)
        if case["mode"] == 0:
            total["flops"] += head
            total["bytes"] += esz * w.d_model * (sum(w.T) + w.d_model)
        else:                # L - 1 levels of `beam` tokens a request, in L - 1 passes (one with an accepted tree)
            passes = 1 if case["drafts"] == "tree" else w.L - 1
            tokens = w.batch * w.beam * (w.L - 1)
            total["flops"] += tokens * (w.n_layers * (2.0 * layer + 4.0 * hq * (ctx + w.L / 2)) + 2.0 * w.d_model * w.T[-1])
            total["bytes"] += passes * esz * (w.n_layers * (layer + 2.0 * w.batch * ctx * hkv) + w.d_model * w.T[-1])
        total["bytes"] += w.batch * w.beam * 4.0 * (w.L + 1)
    return total


def tolerance(case):
    """About four times what the library's own kernels differ by when they sum in another order (the mma.sync attention in
    place of the tcgen05 one, the general GEMM in place of the weight-streaming one) over the shapes and draws of this file."""
    if case["op"] in ("contains", "build"):
        return "exact"
    if _workload(case).dtype == "fp32":
        return {"rel": 1e-5}
    if case["op"] == "prefill":      # hidden states after bf16 layers: 0.0005 (small), 0.0022 (16 layers), 0.0059 (the 7B shape)
        return {"rel": 2.4e-2 if case["shape"] == "7b" else 1e-2, "max": 0.12}
    if case["mode"] == 0:            # 0.0007
        return {"rel": 3e-3, "max": 1e-2}
    return {"rel": 8e-3, "max": 0.12}     # 0.0001 to 0.0017; 0.027 on one score, where two prefixes that tie change places
