"""What the one-launch forward computes in fp32, against 64 bits: one layer, stage by stage.  Every stage is compared with the
same stage computed from the device's own rows in front of it where that isolates it; keys and values are the device's own
bf16 rows, so their rounding plays no part.  The errors are 2-norms relative to the stage's own."""
import math

import pytest
import torch

import mtad_synth as S
import paper_2407_09722_b200 as M
from paper_2407_09722_b200.runtime import DeviceModel

pytestmark = pytest.mark.gpu


def _rms(x, gain, eps):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + eps) * gain.double()


def _rope(x, pos, base):
    half = x.shape[-1] // 2
    ang = pos.double()[:, None] * float(base) ** (-torch.arange(half, dtype=torch.float64, device="cuda") / half)[None]
    c, s = ang.cos()[:, None], ang.sin()[:, None]
    return torch.cat([x[..., :half] * c - x[..., half:] * s, x[..., half:] * c + x[..., :half] * s], -1)


def _error(got, want):
    return ((got.double() - want).norm() / want.norm()).item()


def _layer_errors(sh, batch, rows, length, tree):
    """{stage: error} of one call of batch x rows rows (a chain, or a tree given as (depth, width, keep))."""
    assert sh.layers == 1
    dm = DeviceModel(sh, batch, rows - 1, length + rows + 8)
    trees = [S.beam_tree(*tree, sh.vocab, stream=40 + b) if tree else S.chain_tree(rows - 1, sh.vocab, stream=40 + b)
             for b in range(batch)]
    seqs, T, n = list(range(batch)), batch * rows, rows - 1
    for b in seqs:
        dm.inject(b, length)
        dm.ctx.mtad_seq_set(b, length, 3 + b)
    depth = tree[0] if tree else n
    i32 = dict(dtype=torch.int32, device="cuda")
    tok = torch.tensor([t.tok for t in trees], **i32)
    ref = torch.tensor([t.logq_ref for t in trees], dtype=torch.float32, device="cuda")
    u, res = S.bonus_uniforms(7, rows, batch, sh.vocab, "cuda"), M.ResultBuffers(batch, n, depth)
    if tree:
        par = torch.tensor([t.parent for t in trees], **i32)
        dm.ctx.mtad_verify_tree(seqs, None, n, depth, tok, par, ref, -1.0, u, res)
    else:
        dm.ctx.mtad_verify_chain(seqs, n, tok, ref, -1.0, u, res)
    assert res.status.tolist() == [0] * batch

    terms = 3 if T <= 32 else 2

    def operand_rows(name, k):
        return dm.ctx.region(name, torch.bfloat16)[:T * terms * k].view(T, terms, k).double().sum(1)

    w = {k: v.double() for k, v in dm.weights["layers"][0].items()}
    tokens = torch.tensor([[3 + b] + t.tok for b, t in enumerate(trees)], device="cuda").view(-1)
    pos = length + torch.tensor([[0] + list(t.depth) for t in trees], device="cuda").view(-1)
    h = dm.weights["embed"][tokens].double()
    q = _rope((_rms(h, w["attn_norm"], sh.rms_eps) @ w["wq"].T).view(T, sh.n_q_heads, sh.head_dim), pos, sh.rope_base)
    o = torch.empty_like(q)
    for b, t in enumerate(trees):
        vis = torch.zeros(rows, length + rows, dtype=torch.bool, device="cuda")
        vis[:, :length] = True
        for r in range(rows):
            if r:
                vis[r] |= vis[t.parent[r - 1] + 1]
            vis[r, length + r] = True
        K, V = (dm.cache[0, b, kv, :, :length + rows].double().repeat_interleave(sh.n_q_heads // sh.n_kv_heads, 0)
                for kv in (0, 1))
        s = torch.einsum("rhd,hsd->hrs", q[b * rows:(b + 1) * rows], K) / math.sqrt(sh.head_dim)
        o[b * rows:(b + 1) * rows] = torch.einsum("hrs,hsd->rhd", s.masked_fill(~vis[None], -math.inf).softmax(-1), V)
    o = o.view(T, -1)
    mid = h + o @ w["wo"].T
    f = _rms(mid, w["ffn_norm"], sh.rms_eps)
    gate = f @ w["w_gate"].T
    act = gate * torch.sigmoid(gate) * (f @ w["w_up"].T)
    dev_act = operand_rows("xf", sh.d_ffn)
    hidden = dm.ctx.region("hidden", torch.float32)[:T * sh.d_model].view(T, sh.d_model)
    out = {"attention": _error(operand_rows("xa", sh.n_q_heads * sh.head_dim), o), "gate_up": _error(dev_act, act),
           "down": _error(hidden, mid + dev_act @ w["w_down"].T)}
    print(sh, batch, rows, out)
    return out


# An accumulator of the tensor core loses 6.9e-8 of its value per 64-element k-block added to it, always toward zero (the LM head
# alone: 4.4e-6 over 64 k-blocks, 5.6e-6 over 80, 8.9e-6 over 128).  SwiGLU of two projections that lose alike loses 2.5
# times that: 5.5e-6 where an accumulator takes half of the 64 k-blocks, 11e-6 where it takes them all.  With the error of
# the rows that come in (4.5e-6; 7e-6 as two bf16 terms, beyond 32 rows) that is 7.2 and 12e-6, 9.0 and 13e-6.  Down, 172
# k-blocks, on the device's own activations: 1.7e-6 where an accumulator takes an eighth of them, as with one row of the
# matrix over eight blocks; 3.2e-6 with a quarter, which is what two bf16 terms may add to (2.2e-6).
@pytest.mark.parametrize("batch,rows,tree", [(1, 1, None), (1, 5, None), (1, 9, None), (3, 6, None), (1, 32, None),
                                             (1, 33, (4, 8, 4)), (1, 41, (4, 10, 2)), (8, 7, None), (1, 57, (4, 14, 2)),
                                             (1, 65, (4, 16, 4)), (1, 71, (7, 10, 2)), (8, 10, None)])
def test_accumulators_take_a_part_of_the_k_range(batch, rows, tree):
    e = _layer_errors(S.ModelShape(1, 4096, 32, 32, 128, 11008, 1000), batch, rows, 300, tree)
    many = batch * rows > 32
    assert e["gate_up"] <= (1.1e-5 if many else 9.5e-6), e
    assert e["down"] <= 2.6e-6, e


# Query rows enter the tensor cores as two bf16 terms, 2.4e-6 off, which moves the attention's output by 1.4e-6 at these sizes;
# probabilities of two terms would add 2.4e-6 (together 2.8e-6), three add nothing.  Beyond 32 rows the output itself is
# stored as two terms, 2.5e-6: 2.9e-6 in all, and 3.7e-6 with probabilities of two terms.
@pytest.mark.parametrize("heads,kv_heads,head_dim,batch,rows,tree", [
    (12, 12, 64, 1, 1, None), (12, 12, 64, 1, 5, None), (6, 6, 128, 1, 8, None), (12, 12, 64, 1, 12, None),
    (6, 6, 128, 1, 16, None), (12, 3, 64, 2, 4, None), (12, 12, 64, 1, 17, None), (12, 3, 64, 3, 7, None),
    (12, 12, 64, 8, 7, None), (12, 12, 64, 1, 33, (4, 8, 4)), (6, 6, 128, 1, 41, (4, 10, 2)), (12, 12, 64, 1, 65, (8, 8, 2)),
    (6, 6, 128, 1, 73, (9, 8, 4)), (12, 12, 64, 8, 10, None), (6, 6, 128, 1, 97, (8, 12, 4))])
def test_probabilities_are_exact(heads, kv_heads, head_dim, batch, rows, tree):
    e = _layer_errors(S.ModelShape(1, 768, heads, kv_heads, head_dim, 1024, 1000), batch, rows, 400, tree)
    assert e["attention"] <= (3.3e-6 if batch * rows > 32 else 2.1e-6), e
