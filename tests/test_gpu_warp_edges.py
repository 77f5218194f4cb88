"""Warped rows where the ranking has its edges: fewer tokens than top-k, one chunk of the vocabulary and its last token
alone, the most chunks, one kept token and the most.  Tolerances as test_gpu_warp.py (decisions within the margin are
counted: every row adds a top-k and a top-p boundary)."""
import pytest

import mtad_synth as S
from paper_2407_09722_b200 import binding as Bn
from tests.parity import GpuModel, SeqCase, ParityStats, compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab,top_k,top_p", [(9, 16, 0.95), (1024, 1, 1.0), (1025, 16, 0.8), (33000, 16, 1.0)])
def test_warp_edges(vocab, top_k, top_p):
    sh = S.ModelShape(2, 64, 2, 2, 32, 96, vocab)
    gm = GpuModel(sh, max_batch=1, max_nodes=8, capacity=96)
    stats = ParityStats()
    for it, L in enumerate([30, 41, 52]):
        gm.inject(0, L)
        tree = S.chain_tree(3, vocab, stream=20 + it)
        compare(gm, [SeqCase(0, L, it, tree)], Bn.log_tau(0.2), S.bonus_uniforms(6, it, 1, vocab, "cuda"), chain=True,
                stats=stats, warp=(top_k, top_p))
    assert stats.ok(tie_cap=2), stats
