"""The speculative-decoding accept rule where its launches have their edges: a vocabulary below and around the chunks of
the last draw, one draft token and as many as a warp has lanes, all accepted and none.  Tolerances as test_gpu_spd.py."""
import numpy as np
import pytest
import torch

import mtad_synth as S
import paper_2407_09722_b200 as M
from oracle import mtad_oracle as O
from tests.parity import GpuModel, LP_TOL, MARGIN

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab,gamma,accept", [(11, 1, 0.01), (17, 3, 0.99), (256, 31, 0.01), (257, 32, 0.01), (4099, 32, 0.5)])
def test_spd_edges(vocab, gamma, accept):
    sh = S.ModelShape(2, 64, 2, 2, 32, 96, vocab)
    gm = GpuModel(sh, max_batch=1, max_nodes=32, capacity=96)
    L, root = 40, 3
    gm.inject(0, L)
    gm.ctx.mtad_seq_set(0, L, root)
    cache = gm.cache_bits(0, L)
    rng = np.random.default_rng(vocab + gamma)
    rows = O.log_softmax(rng.normal(scale=0.02, size=(gamma, vocab))).astype(np.float32)
    tok = rng.integers(0, vocab, size=gamma).tolist()
    u_acc = np.full((1, gamma), accept, np.float32)
    u_res = S.bonus_uniforms(5, gamma, 1, vocab, "cuda")
    res = M.ResultBuffers(1, gamma, gamma)
    gm.ctx.mtad_verify_chain_spd([0], gamma, torch.tensor([tok], dtype=torch.int32, device="cuda"),
                                 torch.tensor(rows[None], device="cuda"), torch.tensor(u_acc, device="cuda"), u_res, res)
    gm.ctx.kv_commit([0], res)
    h = res.host()
    r = O.verify_chain_spd(gm.oracle(), cache, L, root, tok, rows.astype(np.float64), u_acc[0].astype(np.float64),
                           u_res[0].cpu().numpy())
    assert int(h["status"][0]) == 0
    if r.margin_accept < MARGIN or r.margin_bonus_robust <= 0:
        pytest.skip("a decision lies within the margin")
    assert int(h["eta"][0]) == r.eta and int(h["winner"][0]) == r.eta - 1 and int(h["n_out"][0]) == r.eta + 1
    assert h["out_tok"][0, :r.eta + 1].tolist() == r.out_tok and h["path"][0, :r.eta].tolist() == r.path
    assert np.max(np.abs(h["out_lp"][0, :r.eta + 1].numpy() - np.asarray(r.out_lp))) < LP_TOL
