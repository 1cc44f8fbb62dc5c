"""Tree attention where its kernel divides: 1 to 4 tiles of 8 row-head pairs
(w * G up to 32) on the cluster kernel, more on the CUDA cores, both head
sizes, contexts shorter than one CTA's first stage and longer than a ring.
"""
from __future__ import annotations

import pytest

import synth
from synth.workloads import Shape, Workload
from tests.gpu_harness import sample_seqs
from tests.test_gpu_tree import ragged, run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,D,width,batch,ctx", [
    (4, 1, 64, 3, 2, (0, 9)), (4, 1, 64, 4, 3, (100, 700)), (6, 2, 128, 5, 2, (120, 140)), (4, 1, 128, 6, 1, (1500, 1500)),
    (8, 2, 128, 8, 2, (300, 500)), (5, 1, 64, 6, 20, (30, 60)), (5, 1, 64, 7, 1, (200, 200))])
def test_tree_row_head_pairs(hq, hkv, D, width, batch, ctx):
    shape = Shape("tree-pairs", 256, hq, hkv, D, 512, 4000, 4, "bf16", 10000.0)
    w = Workload("tree-pairs", shape, batch, *ctx, 3, 1, 31, gain_sigma=0.1, tree_width=width,
                 tree_nodes=min(16, width + 3 * width * width))
    W, I = synth.make_weights(w), ragged(w, synth.make_round_inputs(w))
    _, _, rep = run_case(w, W, I, sample_seqs(batch, 2))
    assert rep["ids_compared"] >= 1
