"""The time-out path of the one-launch forward, the GEMM kernels and the wide attention: a bounded wait that runs out must
end in MTAD_ST_TIMEOUT for every sequence of the call, the kernels must return normally, kv_commit must leave those
sequences alone, and the next call on the same context must match the oracle again.  The wait is made to run out on the
host's request (copies are left out, so the barrier they would complete is never completed); nothing faults and nothing
hangs."""
import math

import pytest
import torch

import mtad_synth as S
import paper_2407_09722_b200 as M
from paper_2407_09722_b200 import binding as Bn
from tests.parity import GpuModel, SeqCase, ParityStats, compare

pytestmark = pytest.mark.gpu
TINY = S.WORKLOADS["tiny"].target
GQA128 = S.ModelShape(2, 512, 8, 2, 128, 1024, 640)


@pytest.mark.parametrize("gamma", [4, 11])      # 15 and 36 rows: three and two bf16 terms
def test_wait_runs_out_then_context_recovers(gamma):
    _runs_out_then_recovers(TINY, gamma, path=1, left_out=1)


# as a chain of launches: 15 rows take the few-row cluster kernel and (gate / up) the stream-K kernel, 36 the many-row cluster
# kernel; in one launch without keys and values; 84 rows of four query heads per KV head: the wide attention of its own
@pytest.mark.parametrize("shape,gamma,path,left_out", [(TINY, 4, 0, 1), (TINY, 11, 0, 1), (TINY, 4, 1, 2), (TINY, 27, 0, 1),
                                                       (GQA128, 27, 1, 2)])
def test_every_kernel_that_waits(shape, gamma, path, left_out):
    _runs_out_then_recovers(shape, gamma, path, left_out)


def _runs_out_then_recovers(shape, gamma, path, left_out):
    gm = GpuModel(shape, max_batch=3, max_nodes=32, capacity=128)
    gm.ctx.mtad_debug_set_path(path)
    V = shape.vocab
    seqs, L = [0, 1, 2], 20
    for s in seqs:
        gm.inject(s, L)
        gm.ctx.mtad_seq_set(s, L, 3 + s)
    trees = [S.chain_tree(gamma, V, stream=70 + s) for s in seqs]
    tok = torch.tensor([t.tok for t in trees], dtype=torch.int32, device="cuda")
    lq = torch.tensor([t.logq for t in trees], dtype=torch.float32, device="cuda")
    u = S.bonus_uniforms(5, 0, 3, V, "cuda")
    res = M.ResultBuffers(3, gamma, gamma)
    gm.ctx.mtad_debug_set_wait(2000, left_out)
    gm.ctx.mtad_verify_chain(seqs, gamma, tok, lq, math.log(0.1), u, res)
    gm.ctx.kv_commit(seqs, res)
    torch.cuda.synchronize()                      # the kernels came back: no fault, no hang
    h = res.host()
    assert all(int(x) & Bn.MTAD_ST_TIMEOUT for x in h["status"].tolist()), h["status"]
    assert h["n_out"].tolist() == [0, 0, 0]
    for s in seqs:
        assert gm.ctx.mtad_seq_get(s) == (L, 3 + s)        # nothing was committed
    # hook off: the same context verifies correctly again (counters and tensor memory were left clean)
    gm.ctx.mtad_debug_set_wait(0, False)
    stats = ParityStats()
    for it in range(2):
        for s in seqs:
            gm.inject(s, L)
        cases = [SeqCase(s, L, 3 + s, S.chain_tree(gamma, V, stream=80 + 8 * it + s)) for s in seqs]
        compare(gm, cases, math.log(0.3), S.bonus_uniforms(6, it, 3, V, "cuda"), chain=True, stats=stats)
    assert stats.ok() and stats.near_ties <= 2, stats


def test_wait_runs_out_in_a_draft():
    """The verification that follows reports it for every sequence of the draft, nothing is committed, and the next draft's
    verification is fine again."""
    W = S.WORKLOADS["tiny"]
    gamma, beam, L, V = 3, 2, 20, W.target.vocab
    gm = GpuModel(W.target, max_batch=2, max_nodes=16, capacity=128, aux=W.aux, aux_capacity=128)
    seqs, n = [0, 1], gamma * beam
    i32, f32 = dict(dtype=torch.int32, device="cuda"), dict(dtype=torch.float32, device="cuda")
    for s in seqs:
        gm.inject(s, L)
        gm.inject_aux(s, L)
    u, u_draft = S.bonus_uniforms(5, 0, 2, V, "cuda"), S.bonus_uniforms(6, 0, 2 * gamma * beam, V, "cuda").view(2, gamma, beam, V)
    tok, parent, depth = (torch.zeros(2, n, **i32) for _ in range(3))
    logq, ref, best = torch.zeros(2, n, **f32), torch.zeros(2, gamma, **f32), torch.zeros(2, gamma, **i32)
    res = M.ResultBuffers(2, n, gamma)
    for path in (0, 1):
        gm.ctx.mtad_debug_set_path(path)
        for fails in (True, False):
            for s in seqs:
                gm.ctx.mtad_seq_set(s, L, 3 + s)
            gm.ctx.mtad_debug_set_wait(*((2000, True) if fails else (0, False)))
            gm.ctx.mtad_draft(seqs, gamma, beam, u_draft, tok, parent, depth, logq, ref, best)
            gm.ctx.mtad_debug_set_wait(0, False)
            gm.ctx.mtad_verify_tree(seqs, None, n, gamma, tok, parent, ref, math.log(0.1), u, res)
            gm.ctx.kv_commit(seqs, res)
            h = res.host()
            if fails:
                assert all(x & Bn.MTAD_ST_TIMEOUT for x in h["status"].tolist()) and h["n_out"].tolist() == [0, 0]
                assert [gm.ctx.mtad_seq_get(s) for s in seqs] == [(L, 3), (L, 4)]
            else:
                assert h["status"].tolist() == [0, 0] and min(h["n_out"].tolist()) >= 1
