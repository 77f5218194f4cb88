"""kv_commit on rows that move: any accepted path a caller may hand in, in any order of its nodes, around the number of rows that
a thread holds in registers."""
import random

import pytest
import torch

import mtad_synth as S
import paper_2407_09722_b200 as M
from paper_2407_09722_b200.runtime import DeviceModel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eta,ascending", [(1, True), (2, False), (8, False), (9, True), (9, False), (32, False)])
@pytest.mark.parametrize("layers,kv_heads,hd", [(1, 1, 32), (3, 5, 64), (40, 40, 128)])
def test_accepted_rows_move(layers, kv_heads, hd, eta, ascending):
    B, N, D = 3, 40, 32
    lens = [0, 17, 30]
    dm = DeviceModel(S.ModelShape(layers, 64, kv_heads, kv_heads, hd, 64, 50), B, N, 80)
    i32 = dict(dtype=torch.int32, device="cuda")
    for b in range(B):
        dm.inject(b, lens[b])
        dm.ctx.mtad_seq_set(b, lens[b], 3)
    tok, n = torch.zeros(B, N, **i32), torch.full((B,), N, **i32)
    parent = torch.tensor([[i - 1 if i < D else -1 for i in range(N)]] * B, **i32)
    res = M.ResultBuffers(B, N, D)
    dm.ctx.mtad_verify_tree(list(range(B)), n, N, D, tok, parent, torch.zeros(B, D, device="cuda"), -1.0,
                            S.bonus_uniforms(7, 1, B, 50, "cuda"), res)
    assert res.status.tolist() == [0] * B
    rng = random.Random(eta + layers)
    paths = [rng.sample(range(N), eta) for _ in range(B)]
    paths = [sorted(p) if ascending else p for p in paths]
    etas = [eta, 0, eta]                                       # (the second sequence keeps its root only)
    want = dm.cache.clone()
    for b in (0, 2):
        for i, node in enumerate(paths[b]):
            want[:, b, :, :, lens[b] + 1 + i] = dm.cache[:, b, :, :, lens[b] + 1 + node]
    res.eta.copy_(torch.tensor(etas, **i32))
    res.path[:, :eta].copy_(torch.tensor(paths, **i32))
    res.out_tok.fill_(7)
    dm.ctx.kv_commit(list(range(B)), res)
    assert res.status.tolist() == [0] * B
    assert [dm.ctx.mtad_seq_get(b) for b in range(B)] == [(lens[b] + etas[b] + 1, 7) for b in range(B)]
    assert torch.equal(dm.cache.view(torch.int16), want.view(torch.int16))
