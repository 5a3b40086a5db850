"""The workloads that performance work on this library is measured on.

A serving program holds the speculator's weights behind a handle, keeps its workspaces and result tensors, and calls
the library between two forward passes of the base model.  Three kinds of pass (`op`):

  step    the base model has scored the candidates: verify them, gather the next context state, draft the next
          candidates (spec_verify -> spec_next_ctx -> spec_draft)
  draft   the draft alone (first call of a sequence; programs that verify elsewhere)
  verify  the verification alone (the last call of a sequence; programs that draft elsewhere)

`B` sequences, `topk` the branching factors of the heads (comma-separated), `K` candidates kept per sequence, `logits`
the type of the base model's logits, `early` the form of verify that stops at a candidate's first mismatch, `e4m3`
heads with the reduced-precision copies attached, `plant` how often the base model agrees with the candidates
(synth.make_base_logits).
"""
import math

import torch

from paper_2404_19124_b200 import binding as spec
from paper_2404_19124_b200 import synth


def _case(name, op, B, topk, K, V, d_base, d_inner, logits="bf16", early=False, e4m3=False, plant="none"):
    c = {"op": op, "B": B, "topk": topk, "K": K, "V": V, "d_base": d_base, "d_inner": d_inner, "logits": logits,
         "early": early, "e4m3": e4m3, "plant": plant}
    return c if name is None else {"name": name, **c}


def _preset(name, preset, **changes):
    p = synth.CONFIGS[preset]
    shape = dict(op="step", B=p.B, topk=",".join(map(str, p.topk)), K=p.K, V=p.V, d_base=p.d_base, d_inner=p.d_inner,
                 plant=p.plant)
    shape.update(changes)
    return _case(name, **shape)


def listed():
    return [
        # The smallest call: launches and host time.  A toy or distilled speculator, a unit test, a smoke run.
        _preset("step_tiny", "tiny"),
        # The repository's production shapes, small batch to large batch and vocabulary: one whole decoding step.
        _preset("step_7b", "llama2-7b"),
        _preset("step_13b", "llama2-13b"),
        _preset("step_34b", "codellama-34b"),
        _preset("step_8b_large_vocab", "llama3-8b"),
        # Batch size 1, the latency case: a few candidates for one sequence ...
        _preset("draft_b1_k5", "llama2-7b", op="draft", B=1, K=5),
        # ... and the single-candidate chain (K = 1), for one sequence and under load.
        _preset("draft_chain_b1", "llama2-13b", op="draft", B=1, topk="1,1,1", K=1),
        _preset("draft_chain_b64", "codellama-34b", op="draft", B=64, topk="1,1,1,1", K=1),
        # The e4m3 copies of the heads, for programs that can spare the memory.
        _preset("step_13b_e4m3", "llama2-13b", e4m3=True),
        # Nothing is a round number: a vocabulary with a few added tokens, widths off the tile sizes.
        _case("step_ragged", "step", B=5, topk="5,3,2", K=11, V=32003, d_base=2568, d_inner=2056, plant="prefix"),
        # Verification alone: fp32 logits, and the early-exit form on a large vocabulary.
        _preset("verify_f32", "llama2-7b", op="verify", logits="f32", plant="bernoulli40"),
        _case("verify_early", "verify", B=16, topk="6,4,3", K=32, V=128256, d_base=4096, d_inner=3072, early=True,
              plant="prefix"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.5)))))))


def draw(rng):
    top = {"bytes": 0.0, "flops": 0.0}
    for c in listed():
        w = work(c)
        top = {k: max(top[k], w[k]) for k in top}
    while True:
        op = rng.choice(["step", "step", "draft", "draft", "verify"])
        n = rng.randint(1, 5)
        topk = [1] * n if rng.random() < 0.25 else [rng.randint(1, 8) for _ in range(n)]
        leaves = math.prod(topk)
        B = _log_int(rng, 1, 64)
        K = _log_int(rng, 1, min(leaves, 64))
        V = _log_int(rng, 1000, 128256)
        e4m3 = op != "verify" and rng.random() < 0.2
        unit = 16 if e4m3 else 8
        d_inner = unit * _log_int(rng, 256 // unit, 4096 // unit)
        d_base = 8 * _log_int(rng, 32, 1024)
        c = _case(None, op, B, ",".join(map(str, topk)), K, V, d_base, d_inner,
                  logits="f32" if op != "draft" and rng.random() < 0.2 else "bf16",
                  early=op != "draft" and rng.random() < 0.25, e4m3=e4m3,
                  plant=rng.choice(["none", "bernoulli40", "prefix"]))
        w = work(c)
        # (the tables of all heads stay resident as well as the logits; no more of either than the largest case has)
        resident = 4.0 * n * V * d_inner if op != "verify" else 0.0
        if leaves <= 4096 and B * leaves <= 6144 and resident <= 6.4e9 and all(w[k] <= top[k] for k in top):
            return c


def _topk(case):
    return tuple(int(t) for t in case["topk"].split(","))


def _trained_like(w, seed, dev):
    """Gives random heads the peaked predictions that a trained speculator makes: every token has eight likely
    successors per head, with logits of 3 to 18 above the rest's spread of 0.6 (the best one gets a few percent to nearly
    all of the probability).  A head row then holds, beside its random part, the embeddings of the tokens that it tends
    to follow; the state of a node correlates with its token's embedding through the mix."""
    g = torch.Generator(device=dev).manual_seed(6000 + seed)
    V, d = w.cfg.V, w.cfg.d_inner
    overlap = 0.5 * math.sqrt((1.0 - w.state_weight ** 2) * d)      # mean of <embedding, state> of a token's own node
    for l in range(w.cfg.n):
        for j in range(8):
            follows = torch.randperm(V, generator=g, device=dev)
            pull = (12.0 * 0.9 ** j / overlap) * (0.5 + torch.rand((V, 1), generator=g, device=dev))
            w.head[l].addcmul_(w.emb[l][follows], pull.to(torch.bfloat16))
    return w


def prepare(case, seed):
    dev = "cuda"
    cfg = synth.SpecConfig("case", case["d_base"], case["d_inner"], case["V"], _topk(case), case["K"], case["B"], None,
                           2.0, case["plant"], seed)
    B, K, n = cfg.B, cfg.K, cfg.n
    s = {"op": case["op"], "topk": cfg.topk, "K": K, "early": case["early"]}
    words = lambda *shape: torch.zeros(shape, dtype=torch.int32, device=dev)
    if s["op"] != "verify":
        s["handle"] = spec.spec_create(_trained_like(synth.make_weights(cfg, device=dev), seed, dev))
        if case["e4m3"]:
            spec.spec_attach_fp8_heads(s["handle"])
        s["ctx"], s["tok"] = synth.make_draft_inputs(cfg, device=dev)
        s["draft_out"] = (words(B, K, n), torch.zeros((B, K), dtype=torch.float32, device=dev))
        need = spec.spec_draft_workspace_bytes(s["handle"], B, cfg.topk, K)
        s["draft_ws"] = torch.empty(need, dtype=torch.uint8, device=dev)
    if s["op"] != "draft":
        bf16 = case["logits"] == "bf16"
        s["cand"] = synth.random_cand_tok(cfg, device=dev)
        s["logits"] = synth.make_base_logits(cfg, s["cand"], device=dev, dtype=torch.bfloat16 if bf16 else torch.float32)
        s["verify_out"] = (words(B), words(B), words(B))
        need = spec.spec_verify_workspace_bytes(B, K, n, cfg.V, spec.SPEC_BF16 if bf16 else spec.SPEC_F32)
        s["verify_ws"] = torch.empty(need, dtype=torch.uint8, device=dev)
    if s["op"] == "step":
        g = torch.Generator(device=dev).manual_seed(5000 + seed)
        s["base_state"] = torch.randn((B, K, n + 1, cfg.d_base), generator=g, device=dev).to(torch.bfloat16)
    return s


def run(s):
    out = {}
    if s["op"] != "draft":
        acc, best, nxt = s["verify_out"]
        spec.spec_verify(s["cand"], s["logits"], accept_len=acc, best_cand=best, next_tok=nxt, workspace=s["verify_ws"],
                         early_exit=s["early"])
        out.update(accept_len=acc, best_cand=best, next_tok=nxt)
    if s["op"] == "verify":
        return out
    ctx, tok = s["ctx"], s["tok"]
    if s["op"] == "step":
        spec.spec_next_ctx(s["base_state"], best, acc, ctx_state=ctx, err_workspace=s["verify_ws"])
        tok = nxt
        out["ctx_state"] = ctx
    cand, logp = s["draft_out"]
    spec.spec_draft(s["handle"], ctx, tok, s["topk"], s["K"], cand_tok=cand, cand_logp=logp, workspace=s["draft_ws"])
    out.update(cand_tok=cand, cand_logp=logp)
    return out


def work(case):
    """Weights, gathered embedding rows, logits and results once each; the multiply-adds of the two matrices of a head."""
    topk, B, K, V, d = _topk(case), case["B"], case["K"], case["V"], case["d_inner"]
    n, size, flops = len(topk), 0.0, 0.0
    if case["op"] != "verify":
        rows = B
        for l, k in enumerate(topk):
            parents, d_in = (B, case["d_base"]) if l == 0 else (rows // topk[l - 1], d)
            size += 2.0 * d * d_in + 2.0 * min(rows, V) * d + 8.0 * d
            if case["e4m3"] and rows <= 128:      # the copy, its scales, and the rows whose logits are recomputed
                size += 1.0 * V * d + 4.0 * V + 2.0 * rows * k * d
            else:
                size += 2.0 * V * d
            flops += 2.0 * parents * d * d_in + 2.0 * rows * V * d
            rows *= k
        size += B * (2.0 * case["d_base"] + 4.0) + B * K * (4.0 * n + 4.0)
    if case["op"] != "draft":
        # early exit: rows up to the first mismatch, by how the matches are planted
        rows = n + 1.0
        if case["early"]:
            rows = {"none": 1.0, "bernoulli40": (1 - 0.4 ** (n + 1)) / 0.6, "prefix": n / 2.0 + 1}[case["plant"]]
        size += B * K * (rows * V * (2.0 if case["logits"] == "bf16" else 4.0) + 4.0 * n) + 12.0 * B
    if case["op"] == "step":
        size += 4.0 * B * case["d_base"]
    return {"bytes": size, "flops": flops}


def tolerance(case):
    if case["op"] == "verify":
        return "exact"
    # cand_logp is a sum of fp32 log-softmax values of logits whose states are rounded to bf16; cand_tok changes where
    # two candidates' scores are closer than that.
    return {"rel": 1e-3, "max": 1e-2, "differ": 0.01}
