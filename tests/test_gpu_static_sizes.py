"""What fits the fixed scratch array of mtad_verify_chain_static: shapes and chain lengths whose step as a chain of launches
fits are accepted, whether or not the arrays of the one-launch forward fit beside it, and give what an ordinary context
gives (tolerance as in test_zz_no_alloc.py)."""
import math

import pytest
import torch

import mtad_synth as S
import paper_2407_09722_b200 as M
from paper_2407_09722_b200 import binding as Bn
from paper_2407_09722_b200.runtime import DeviceModel

pytestmark = pytest.mark.gpu
LP_TOL = 2e-3


@pytest.mark.parametrize("shape,gamma,capacity,both_fit", [
    (S.ModelShape(2, 256, 4, 4, 64, 688, 32000), 1, 64, True),
    (S.ModelShape(2, 256, 4, 4, 64, 688, 32000), 8, 128, True),
    (S.ModelShape(4, 512, 8, 8, 64, 1376, 32000), 4, 128, True),
    (S.ModelShape(2, 512, 8, 8, 64, 1376, 1024), 32, 8192, True),
    (S.ModelShape(2, 512, 8, 8, 64, 1376, 32000), 7, 8192, False),
    (S.ModelShape(4, 512, 4, 4, 128, 2048, 32000), 8, 128, False),
])
def test_accepted_sizes(shape, gamma, capacity, both_fit):
    dm = DeviceModel(shape, max_batch=1, max_nodes=gamma, capacity=capacity)
    assert (dm.ctx.workspace_bytes <= Bn.MTAD_STATIC_SCRATCH_BYTES) == both_fit, dm.ctx.workspace_bytes
    L, V = 50, shape.vocab
    tree = S.chain_tree(gamma, V, stream=31)
    tok = torch.tensor(tree.tok, dtype=torch.int32, device="cuda")
    lq = torch.tensor(tree.logq, dtype=torch.float32, device="cuda")
    u = S.bonus_uniforms(3, gamma, 1, V, "cuda")
    dm.inject(0, L)
    want, got = M.ResultBuffers(1, gamma, gamma), M.ResultBuffers(1, gamma, gamma)
    dm.ctx.mtad_seq_set(0, L, 7)
    dm.ctx.mtad_verify_chain([0], gamma, tok, lq, math.log(0.1), u, want)
    assert Bn.mtad_verify_chain_static(dm.desc, L, 7, gamma, tok, lq, math.log(0.1), u, got) == Bn.MTAD_OK
    w, g = want.host(), got.host()
    assert int(w["status"][0]) == 0 and int(g["status"][0]) == 0
    for k in ("node_lp", "node_LP", "row_lse"):
        assert torch.max(torch.abs(g[k] - w[k])).item() <= LP_TOL, k
    if w["margin"].min().item() > 1e-3:
        assert int(g["eta"][0]) == int(w["eta"][0])
