"""Sums of squares of a row, whose root divides everything that follows, on rows made to lose where a sum is a long chain: one
element of 4096 (2^24 squared, where fp32 steps by 2) beside many whose squares, 0.9, a running sum of 2^24 does not take in."""
import math

import pytest
import torch

import mtad_synth as S
import paper_2407_09722_b200 as M
from paper_2407_09722_b200.runtime import DeviceModel

pytestmark = pytest.mark.gpu
BIG, SMALL = 4096.0, 0.94921875


def _column(w):
    """Only the first input feature counts: every output is one product, which no accumulator rounds."""
    w[:, 1:] = 0
    w[:, 0] = torch.linspace(0.5, 1.5, w.shape[0], device="cuda") / 64
    return w[:, 0].double()


def test_parts_of_a_row():
    """The parts of a row that the blocks of a projection leave, a small element in each but the first.  Added a lane per part in five
    rounds and a tree, their sum is 1.4e-7 off; in runs of 16 parts one after the other 9.7e-7.  SwiGLU carries about as much into
    its outputs, and rounding them to two bf16 terms leaves 5e-8 of their mean."""
    sh = S.ModelShape(1, 4096, 8, 8, 64, 8192, 200)
    dm = DeviceModel(sh, 8, 4, 40)
    layer, tile = dm.weights["layers"][0], 32                  # features of a block: 4096 over 148, in eights
    dm.weights["embed"].zero_()[:, ::tile] = SMALL
    dm.weights["embed"][:, 0] = BIG
    layer["wo"].zero_()
    layer["ffn_norm"].fill_(1.0)
    gate, up = _column(layer["w_gate"]), _column(layer["w_up"])
    for b in range(8):
        dm.inject(b, 16)
        dm.ctx.mtad_seq_set(b, 16, 3)
    tok = torch.tensor([S.chain_tree(4, sh.vocab, stream=b).tok for b in range(8)], dtype=torch.int32, device="cuda")
    res = M.ResultBuffers(8, 4, 4)
    dm.ctx.mtad_verify_chain(list(range(8)), 4, tok, torch.zeros(8, 4, device="cuda"), -1.0,
                             S.bonus_uniforms(7, 1, 8, sh.vocab, "cuda"), res)
    assert res.status.tolist() == [0] * 8
    act = dm.ctx.region("xf", torch.bfloat16)[:40 * 2 * sh.d_ffn].view(40, 2, sh.d_ffn).double().sum(1)
    x = BIG / math.sqrt((BIG ** 2 + (sh.d_model // tile - 1) * SMALL ** 2) / sh.d_model + sh.rms_eps)
    want = gate * x * torch.sigmoid(gate * x) * (up * x)
    off = (act / want - 1).mean(1).abs().max().item()
    print(off)
    assert off < 4e-7


def test_rows_of_a_draft():
    """The embedding rows that the selection of a draft step makes for the next, a small element in every second place.  Added by
    128 threads and a tree the sum is 8e-7 off, by a warp of which each lane keeps one sum 3.4e-6; its root scales the queries,
    whose rounding to 16 bits and more leaves 1e-7 of their mean."""
    target, sh = S.ModelShape(1, 128, 2, 2, 64, 344, 200), S.ModelShape(1, 4096, 16, 16, 128, 512, 200)
    gamma, b, length = 2, 4, 4
    dm = DeviceModel(target, 1, gamma * b, 64, aux=sh, aux_capacity=64)
    layer = dm.aux_weights["layers"][0]
    dm.aux_weights["embed"].zero_()[:, ::2] = SMALL
    dm.aux_weights["embed"][:, 0] = BIG
    layer["attn_norm"].fill_(1.0)
    w = _column(layer["wq"]).view(sh.n_q_heads, 2, 64)
    dm.ctx.mtad_seq_set(0, length, 3, aux_len=length)
    i32, f32 = dict(dtype=torch.int32, device="cuda"), dict(dtype=torch.float32, device="cuda")
    tok, parent, depth = (torch.zeros(1, gamma * b, **i32) for _ in range(3))
    dm.ctx.mtad_draft([0], gamma, b, S.uniforms(0, 37, gamma * b * sh.vocab, "cuda").view(1, gamma, b, sh.vocab), tok, parent, depth,
                      torch.zeros(1, gamma * b, **f32), torch.zeros(1, gamma, **f32), torch.zeros(1, gamma, **i32),
                      n_nodes=torch.zeros(1, **i32))
    q = sum(dm.ctx.region(n, torch.bfloat16)[:b * 2048].view(b, sh.n_q_heads, 2, 64).double() for n in ("q_hi", "q_lo"))
    angle = (length + 1) * float(sh.rope_base) ** (-torch.arange(64, dtype=torch.float64, device="cuda") / 64)
    x = BIG / math.sqrt((BIG ** 2 + (sh.d_model // 2 - 1) * SMALL ** 2) / sh.d_model + sh.rms_eps)
    y = w * x * math.log2(math.e) / math.sqrt(sh.head_dim)
    want = torch.stack([y[:, 0] * angle.cos() - y[:, 1] * angle.sin(), y[:, 1] * angle.cos() + y[:, 0] * angle.sin()], 1)
    off = (((q * want).sum((1, 2, 3)) / (want * want).sum()) - 1).abs().max().item()
    print(off)
    assert off < 1e-6
