"""A device, or a part of one, that cannot hold the blocks of the one-launch forward at once: its calls, and those whose
attention alone is such a launch, run as a chain of launches with the attention of mma.sync warps, whether that is known
when the context is made or the driver refuses the launch later.  Compared with the CPU oracle at the edges of that
attention's variants (query rows per KV head: a packed tile, one, two, up to four, five and more tiles of 16)."""
import threading

import pytest
import torch

import mtad_synth as S
import paper_2407_09722_b200 as M
from paper_2407_09722_b200 import binding as Bn
from tests.parity import GpuModel, SeqCase, ParityStats, compare

pytestmark = pytest.mark.gpu
MHA64 = S.ModelShape(2, 256, 4, 4, 64, 688, 1000)
GQA128 = S.ModelShape(2, 512, 8, 2, 128, 1024, 640)              # four query rows of a KV head per row of a call


def _compare(gm, rows, tree, lengths, it=0):
    sh, stats, cases = gm.shape, ParityStats(), []
    for b, L in enumerate(lengths):
        gm.inject(b, L)
        t = S.beam_tree(*tree, sh.vocab, stream=270 + b) if tree else S.chain_tree(rows - 1, sh.vocab, stream=250 + b)
        assert len(t.tok) == rows - 1
        cases.append(SeqCase(b, L, int(S.token_ids(9, (23 << 40) | b, 1, sh.vocab)[0]), t))
    compare(gm, cases, Bn.log_tau(0.3), S.bonus_uniforms(9, rows + it, len(lengths), sh.vocab, "cuda"), chain=tree is None,
            stats=stats)
    assert stats.ok(), stats


@pytest.mark.parametrize("path", [0, 2])
@pytest.mark.parametrize("shape,rows,tree,lengths", [
    (MHA64, 5, None, [130]), (MHA64, 9, None, [64]), (MHA64, 17, (4, 4, 2), [100]), (MHA64, 33, (4, 8, 4), [65]),
    (MHA64, 71, (7, 10, 2), [129]), (MHA64, 97, (8, 12, 4), [200]), (GQA128, 2, None, [63, 1]), (GQA128, 7, None, [90, 128, 5]),
    (GQA128, 33, (4, 8, 4), [127])])
def test_chain_of_launches(shape, rows, tree, lengths, path):
    gm = GpuModel(shape, max_batch=len(lengths), max_nodes=rows, capacity=320)
    launches = []
    for it, p in enumerate((path, 1)):                           # and back: the plans of the other path are not kept
        gm.ctx.mtad_debug_set_path(p)
        n = Bn.mtad_kernel_launches()
        _compare(gm, rows, tree, lengths, it)
        launches.append(Bn.mtad_kernel_launches() - n)
    assert launches[0] > launches[1] or rows * len(lengths) > 80, launches


@pytest.mark.parametrize("shape,rows,tree,lengths,chain", [
    (S.ModelShape(1, 256, 32, 32, 64, 512, 500), 1, None, [40 + 5 * b for b in range(33)], True),      # 33 sequences
    (S.ModelShape(1, 256, 32, 32, 64, 512, 500), 2, None, [30 + 9 * b for b in range(31)], False),     # 31 x 32 KV heads
    (S.ModelShape(1, 256, 32, 32, 64, 512, 500), 1, None, [64] * 32, True),                            # 32 x 32
    (S.ModelShape(1, 256, 2, 2, 64, 512, 500), 2, None, [20 + b for b in range(32)], True),            # 64 rows of 32
    (S.ModelShape(1, 256, 2, 2, 128, 512, 500), 2, None, [20 + b for b in range(32)], False),          # heads of 128
    (MHA64, 81, (5, 16, 4), [90], True), (MHA64, 97, (8, 12, 4), [90], True),                          # six tiles of 16, seven
    (MHA64, 145, (9, 16, 4), [90], False), (GQA128, 81, (5, 16, 4), [90], False),
])
def test_the_faster_way_is_taken(shape, rows, tree, lengths, chain):
    """Few long calls as one launch (beyond 80 rows: their attention), calls of many sequences with heads of 64 as a chain."""
    gm = GpuModel(shape, max_batch=len(lengths), max_nodes=max(rows - 1, 1), capacity=480)
    launches = []
    for it, path in enumerate((1, 0)):
        gm.ctx.mtad_debug_set_path(path)
        n = Bn.mtad_kernel_launches()
        _compare(gm, rows, tree, lengths, it)
        launches.append(Bn.mtad_kernel_launches() - n)
    assert (launches[0] == launches[1]) == chain, launches



@pytest.mark.parametrize("shape,wide", [(S.ModelShape(2, 256, 2, 2, 128, 512, 500), True), (MHA64, False)])
def test_keys_from_which_the_wide_attention_is_taken(shape, wide):
    """Three tiles of query rows a KV head: mma.sync warps up to 2047 keys, and with heads of 64 beyond them."""
    gm = GpuModel(shape, max_batch=2, max_nodes=40, capacity=2100)
    used = []
    for L in (2006, 2007):
        n = Bn.mtad_kernel_launches()
        _compare(gm, 41, (4, 10, 2), [L, 50], L)
        used.append(Bn.mtad_kernel_launches() - n)
    assert used[0] - used[1] == (shape.layers if wide else 0), used        # (two launches a layer, one)


@pytest.mark.parametrize("shape,rows", [(MHA64, 5), (S.ModelShape(2, 256, 2, 2, 128, 512, 500), 6), (GQA128, 5)])
def test_stale_partials_of_ragged_batches(shape, rows):
    """Beyond 80 rows, few of them per sequence: the attention of mma.sync warps, whose splits past a short sequence's keys are
    empty.  What earlier calls left in their partials must not matter, a NaN neither."""
    lengths = [0, 250, 1, 64, 63, 190, 7, 128, 33, 3, 255, 70, 100, 0, 129, 20, 200]
    gm = GpuModel(shape, max_batch=len(lengths), max_nodes=rows, capacity=320)
    for it in range(2):
        gm.ctx.region("attn_part", torch.float32).fill_(float("nan"))
        _compare(gm, rows, None, lengths, it)


def _chain_call(gm, L, gamma, seed):
    t, V = S.chain_tree(gamma, gm.shape.vocab, stream=seed), gm.shape.vocab
    gm.inject(0, L)
    gm.ctx.mtad_seq_set(0, L, 3)
    tok = torch.tensor([t.tok], dtype=torch.int32, device="cuda")
    lq = torch.tensor([t.logq], dtype=torch.float32, device="cuda")
    res, u = M.ResultBuffers(1, gamma, gamma), S.bonus_uniforms(9, seed, 1, V, "cuda")
    return res, lambda stream=None: gm.ctx.mtad_verify_chain([0], gamma, tok, lq, Bn.log_tau(0.3), u, res, stream=stream)


def _same(a, b):
    return all(torch.equal(a[k], b[k]) for k in ("eta", "winner", "n_out", "out_tok", "out_lp", "node_lp", "row_lse", "status"))


@pytest.mark.parametrize("gamma,path", [(4, 1), (4, 0), (30, 1)])
def test_capture(gamma, path):
    """A verification recorded in a CUDA graph and replayed gives what the call gives."""
    gm = GpuModel(MHA64, max_batch=1, max_nodes=32, capacity=320)
    gm.ctx.mtad_debug_set_path(path)
    res, call = _chain_call(gm, 150, gamma, 3)
    call()
    torch.cuda.synchronize()
    want = res.host()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    for _ in range(2):
        res.buf.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert _same(res.host(), want)
    del graph


def test_two_contexts_on_two_streams():
    """Calls of two contexts, each on its own stream and thread: what one of them waits for never depends on the other."""
    made = []
    for k, sh in enumerate((MHA64, GQA128)):
        gm = GpuModel(sh, max_batch=1, max_nodes=32, capacity=320)
        res, call = _chain_call(gm, 140 + 20 * k, 8 + 16 * k, 5 + k)
        call()
        torch.cuda.synchronize()
        made.append((gm, res, call, res.host(), torch.cuda.Stream()))

    def work(k):
        for _ in range(40):
            made[k][2](made[k][4])

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for gm, res, call, want, _ in made:
        assert _same(res.host(), want)
