"""GPU parity of rounds with more activation rows than one tile of the
streamed projections holds: 256 rows (128 for gate/up, 64 for the LM head's
top-k lists).  Such rows are cut into tiles, each multiplied with the same
weights: a prompt's prefill, a batch whose sequences each bring several
accepted tokens, and batches and trees of more than 64 rows at the LM head.
"""
from __future__ import annotations

from dataclasses import replace

import pytest

import synth
from synth.workloads import Workload
from tests.gpu_harness import sample_seqs
from tests.test_gpu_ragged_vocab import TINY_V4000
from tests.test_gpu_round import _check
from tests.test_gpu_tree import ragged, run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,n_new,topk", [(1, 256, 1), (1, 257, 1), (3, 129, 8), (1, 1030, 1), (65, 6, 8), (129, 1, 1),
                                              (130, 2, 3)])
def test_rows_beyond_one_tile(batch, n_new, topk):
    w = Workload("row-tiles", TINY_V4000, batch, 8, 40, n_new, topk, 11)
    W, I = synth.make_weights(w), synth.make_round_inputs(w)
    _, _, rep = _check(w, W, ragged(w, I), sample_seqs(batch, 3), topk=topk)
    assert rep["ids_compared"] >= 1


def test_tree_rows_beyond_one_tile():
    """33 sequences of a width-4 tree: 132 rows per step, three row tiles at the LM head."""
    w = Workload("row-tiles-tree", replace(TINY_V4000, name="tiny-v4000-k3", n_steps=3), 33, 8, 40, 2, 1, 12,
                 gain_sigma=0.1, tree_width=4, tree_nodes=10)
    W, I = synth.make_weights(w), ragged(w, synth.make_round_inputs(w))
    _, _, rep = run_case(w, W, I, sample_seqs(33, 3))
    assert rep["ids_compared"] >= 1
