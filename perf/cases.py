"""The calls a decoding program makes into this library, as timed cases: verification steps on draft chains and
candidate trees, the speculative-decoding accept rule, warped rows, prompt chunks, drafts, and whole iterations
(draft, verification, cache roll-forward).

Shapes are the workloads of `mtad_synth` (the benchmark's and the tests'); the 70B-shaped target runs with eight of its
layers, as in the tests, so that several states fit one GPU.  Weights, caches, draft tokens, draft likelihoods and
uniforms are random with the workloads' distributions and depend on the seed alone.
"""
from __future__ import annotations

import dataclasses
import math

import torch

import mtad_synth as S
import paper_2407_09722_b200 as M

LOG_TAU = math.log(0.1)

# name -> (target shape, auxiliary shape)
MODELS = {
    "tiny": (S.WORKLOADS["tiny"].target, S.WORKLOADS["tiny"].aux),
    "7b": (S.WORKLOADS["7b_chain"].target, S.WORKLOADS["7b_chain"].aux),
    "13b": (S.WORKLOADS["13b_batched_chain"].target, S.WORKLOADS["13b_batched_chain"].aux),
    "70b_8l": (dataclasses.replace(S.WORKLOADS["70b_gqa_tree"].target, layers=8), S.WORKLOADS["70b_gqa_tree"].aux),
}

# op:  chain      verify_chain + kv_commit
#      chain_spd  verify_chain_spd + kv_commit (vanilla speculative decoding on the same forward)
#      prompt     verify_chain that accepts every token (tau = 0) + kv_commit: how a prompt enters the cache
#      tree       verify_tree + kv_commit
#      draft      mtad_draft alone
#      iteration  mtad_draft, verification of its output sequence as a chain, kv_commit of both caches
#      mmtad      mtad_draft that keeps every candidate, verification of that tree, kv_commit of both caches
_DEFAULTS = {"batch": 1, "beam": 4, "width": 0, "keep": 0, "top_k": 0, "top_p": 1.0}


def _case(name, model, op, gamma, kv_lo, kv_hi, **more):
    c = dict(_DEFAULTS, model=model, op=op, gamma=gamma, kv_lo=kv_lo, kv_hi=kv_hi)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # smallest calls: one decode iteration of the tiny pair, launches and latency only
        _case("tiny_iteration", "tiny", "iteration", 4, 32, 32),
        # the auxiliary model's share of an iteration: one sequence, and a batch of eight
        _case("7b_pair_draft", "7b", "draft", 4, 2048, 2048),
        _case("13b_pair_draft_batch8", "13b", "draft", 6, 1024, 3072, batch=8),
        # the ordinary decode step: a chain of four tokens against 2048 committed ones
        _case("7b_chain", "7b", "chain", 4, 2048, 2048),
        # the same on warped rows (top-k 10, top-p 0.9), at an odd length and another chain length
        _case("7b_chain_warped", "7b", "chain", 6, 1531, 1531, top_k=10, top_p=0.9),
        # three ragged sequences under the speculative-decoding rule
        _case("7b_spd_batch3", "7b", "chain_spd", 5, 333, 2222, batch=3),
        # a chunk in the middle of a 512-token prompt
        _case("7b_prompt_chunk", "7b", "prompt", 32, 231, 231),
        # candidate tree of 4 layers x 16 nodes
        _case("7b_tree64", "7b", "tree", 4, 2048, 2048, width=16, keep=4),
        # multi-candidate decoding as a whole: drafted 64-node tree, verification, both caches rolled forward
        _case("7b_mmtad_iteration", "7b", "mmtad", 4, 1111, 1111),
        # batched serving: eight ragged sequences, chains of six
        _case("13b_chain_batch8", "13b", "chain", 6, 1024, 3072, batch=8),
        # the widest target: grouped-query attention, a tree of 4 layers x 32 nodes
        _case("70b_8l_tree128", "70b_8l", "tree", 4, 1024, 1024, width=32, keep=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    model = rng.choice(["tiny", "7b", "7b", "7b", "13b", "13b", "70b_8l"])
    op = rng.choice(["chain", "chain", "chain_spd", "prompt", "tree", "tree", "draft", "iteration", "mmtad"])
    hi = 400 if model == "tiny" else 2800
    kv_hi = _log_int(rng, 16, hi)
    kv_lo = max(8, int(kv_hi * rng.uniform(0.3, 1.0)))
    max_rows = 72                                     # rows of a call: no drawn case costs more than the listed ones
    more = {}
    if op in ("chain", "chain_spd"):
        gamma = rng.randint(0 if op == "chain" else 1, 8)
        batch = min(8, _log_int(rng, 1, 8), max(1, max_rows // (gamma + 1)))
        more["batch"] = batch
        if op == "chain" and rng.random() < 0.3:
            more.update(top_k=rng.randint(2, 16), top_p=round(rng.uniform(0.5, 1.0), 3))
    elif op == "prompt":
        gamma = rng.randint(8, 32)
        more["batch"] = rng.choice([1, 1, 2])
    elif op == "tree":
        gamma = rng.randint(2, 5)
        keep = rng.randint(1, 4)
        width = keep * rng.randint(1, max(1, min(6, (max_rows - 1) // (gamma * keep))))
        more.update(width=width, keep=keep, batch=2 if 2 * (gamma * width + 1) <= max_rows and rng.random() < 0.3 else 1)
    else:
        gamma = rng.randint(2, 6)
        beam = rng.randint(1, 8 if op != "mmtad" else 4)
        while op == "mmtad" and gamma * beam * beam + 1 > max_rows:
            beam -= 1
        rows = {"draft": beam, "iteration": gamma + 1, "mmtad": gamma * beam * beam + 1}[op]
        more.update(beam=beam, batch=min(_log_int(rng, 1, 8), max(1, max_rows // rows)))
    if more.get("batch", 1) == 1:
        kv_lo = kv_hi
    return _case(None, model, op, gamma, kv_lo, kv_hi, **more)


# ---------------------------------------------------------------------------------------------------------------

def _lengths(case):
    lo, hi, b = case["kv_lo"], case["kv_hi"], case["batch"]
    return [lo + (hi - lo) * ((i * 2654435761 + 40503) % (1 << 16)) // (1 << 16) for i in range(b)]


def _nodes(case):
    if case["op"] == "tree":
        return case["gamma"] * case["width"]
    if case["op"] == "mmtad":
        return case["gamma"] * case["beam"] ** 2
    return case["gamma"]


def _drafts(case):
    return case["op"] in ("draft", "iteration", "mmtad")


def _verifies(case):
    return case["op"] != "draft"


def _weights(shape, gen):
    def mat(*dims):
        return torch.empty(*dims, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=gen)

    def gain(n):
        return torch.empty(n, dtype=torch.bfloat16, device="cuda").normal_(1.0, 0.1, generator=gen)

    return {"embed": mat(shape.vocab, shape.d_model), "lm_head": mat(shape.vocab, shape.d_model),
            "final_norm": gain(shape.d_model),
            "layers": [{n: gain(d[0]) if len(d) == 1 else mat(*d) for n, d in S.layer_tensor_shapes(shape).items()}
                       for _ in range(shape.layers)]}


def _cache(shape, batch, capacity, gen):
    return torch.empty(S.kv_cache_shape(shape, batch, capacity), dtype=torch.bfloat16, device="cuda").normal_(generator=gen)


def _uniforms(gen, *dims):
    return torch.rand(*dims, device="cuda", generator=gen).clamp_(2.0 ** -24, 1.0 - 2.0 ** -24)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    target, aux = MODELS[case["model"]]
    if case["op"] == "draft":                         # the auxiliary model does all the work of this call
        target = dataclasses.replace(target, layers=1)
    B, g, b, N, V = case["batch"], case["gamma"], case["beam"], _nodes(case), target.vocab
    lens = _lengths(case)
    drafted = g * b * b if case["op"] == "mmtad" else g * b
    keep = []
    cache = _cache(target, B, max(lens) + max(N, 1) + 8, gen)
    desc = M.make_desc(target, _weights(target, gen), cache, keep)
    aux_desc = None
    if _drafts(case):
        aux_cache = _cache(aux, B, max(lens) + drafted + 40, gen)
        aux_desc = M.make_desc(aux, _weights(aux, gen), aux_cache, keep)
    ctx = M.Context(desc, aux_desc, B, max(N, drafted if _drafts(case) else N), keep=keep)
    if case["top_k"]:
        ctx.mtad_set_warp(case["top_k"], case["top_p"])
    i32 = dict(dtype=torch.int32, device="cuda")
    f32 = dict(dtype=torch.float32, device="cuda")
    s = {"case": case, "ctx": ctx, "cache": cache, "lens": lens, "seqs": list(range(B)),
         "roots": torch.randint(0, V, (B,), generator=torch.Generator().manual_seed(seed)).tolist(),
         "u": _uniforms(gen, B, V), "res": M.ResultBuffers(B, N, g)}
    if _drafts(case):
        s["draft"] = {"tok": torch.zeros(B, drafted, **i32), "parent": torch.zeros(B, drafted, **i32),
                      "depth": torch.zeros(B, drafted, **i32), "node_logq": torch.zeros(B, drafted, **f32),
                      "logq_ref": torch.zeros(B, g, **f32), "best_path": torch.zeros(B, g, **i32),
                      "n_nodes": torch.zeros(B, **i32)}
        s["u_draft"] = _uniforms(gen, B, g, b, V)
    elif case["op"] == "tree":
        trees = [S.beam_tree(g, case["width"], case["keep"], V, seed, i) for i in range(B)]
        s["tok"] = torch.tensor([t.tok for t in trees], **i32)
        s["parent"] = torch.tensor([t.parent for t in trees], **i32)
        s["logq"] = torch.tensor([t.logq_ref for t in trees], **f32)
        s["n_nodes"] = torch.full((B,), N, **i32)
    elif g:
        trees = [S.chain_tree(g, V, seed, i) for i in range(B)]
        s["tok"] = torch.tensor([t.tok for t in trees], **i32)
        s["logq"] = torch.tensor([t.logq for t in trees], **f32)
        if case["op"] == "chain_spd":
            s["q_rows"] = torch.randn(B, g, V, generator=gen, **f32).log_softmax(-1)
            s["u_accept"] = _uniforms(gen, B, g)
    for i in range(B):
        ctx.mtad_seq_set(i, lens[i], s["roots"][i])
    torch.cuda.synchronize()
    return s


def run(s):
    case, ctx, seqs, res = s["case"], s["ctx"], s["seqs"], s["res"]
    op, g, N = case["op"], case["gamma"], _nodes(case)
    out = {}
    if op != "draft":                                 # every pass starts from the same committed lengths
        for i in seqs:
            ctx.mtad_seq_set(i, s["lens"][i], s["roots"][i])
    if _drafts(case):
        d = s["draft"]
        ctx.mtad_draft(seqs, g, case["beam"], s["u_draft"], d["tok"], d["parent"], d["depth"], d["node_logq"],
                       d["logq_ref"], d["best_path"], keep_all_candidates=op == "mmtad", n_nodes=d["n_nodes"])
        out.update(d)
        if op == "iteration":
            chain = d["tok"].gather(1, d["best_path"].long())
            ctx.mtad_verify_chain(seqs, g, chain, d["logq_ref"], LOG_TAU, s["u"], res)
        elif op == "mmtad":
            ctx.mtad_verify_tree(seqs, d["n_nodes"], N, g, d["tok"], d["parent"], d["logq_ref"], LOG_TAU, s["u"], res)
    elif op == "tree":
        ctx.mtad_verify_tree(seqs, s["n_nodes"], N, g, s["tok"], s["parent"], s["logq"], LOG_TAU, s["u"], res)
    elif op == "chain_spd":
        ctx.mtad_verify_chain_spd(seqs, g, s["tok"], s["q_rows"], s["u_accept"], s["u"], res)
    else:
        ctx.mtad_verify_chain(seqs, g, s.get("tok"), s.get("logq"), -math.inf if op == "prompt" else LOG_TAU, s["u"], res)
    if _verifies(case):
        ctx.kv_commit(seqs, res)
        # what a decode loop consumes, and the cache rows this step left (committed ones first).  The extra-token
        # candidates of rows that were not chosen stay out: each is one draw, and a near tie in any would be a mismatch.
        out.update({n: getattr(res, n) for n in ("eta", "winner", "path", "n_out", "out_tok", "out_lp", "status")})
        if N:
            out["node_lp"] = res.node_lp
            if not case["top_k"] and op != "chain_spd":
                out["node_LP"] = res.node_LP
        out["row_lse"] = res.row_lse
        for i in seqs:
            out["kv%d" % i] = s["cache"][:, i, :, :, s["lens"][i]:s["lens"][i] + N + 1]
    return out


def work(case):
    target, aux = MODELS[case["model"]]
    B, g, b, N = case["batch"], case["gamma"], case["beam"], _nodes(case)
    lens = _lengths(case)
    nbytes = flops = 0.0

    def forward(shape, rows, weights):
        """rows of every sequence through the model; weights: read here (once per pass, however many steps use them)"""
        nonlocal nbytes, flops
        w = shape.layers * shape.layer_params() + shape.vocab * shape.d_model
        flops += 2.0 * w * rows * B + sum(4.0 * rows * (L + rows / 2.0) * shape.q_dim * shape.layers for L in lens)
        if weights:
            nbytes += 2.0 * w + shape.kv_bytes_per_token() * float(sum(lens))
        nbytes += shape.kv_bytes_per_token() * rows * B + 2.0 * rows * B * shape.d_model

    if _drafts(case):
        for step in range(g):
            forward(aux, 1 if step == 0 else b, step == 0)
        nbytes += 4.0 * B * target.vocab * (1 + (g - 1) * b)                 # the uniforms that the selection reads
    if _verifies(case):
        forward(target, N + 1, True)
        nbytes += 4.0 * B * target.vocab * (1 + (g if case["op"] == "chain_spd" else 0))
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Keys and values are rounded to bf16 after the fp32 projection: where two implementations differ in the last fp32
    # bits a few elements land on the neighbouring bf16 value (2^-8 of the value) and carry the difference on.  Measured
    # between the tensor-core and the CUDA-core path over the listed cases: 1.6e-3 and 0.016 on the deepest layers' cache
    # rows, 2e-4 and 1e-3 on log-probabilities, no whole value different.
    return {"rel": 6e-3, "max": 0.06}
