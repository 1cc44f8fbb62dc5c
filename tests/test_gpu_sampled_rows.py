"""Sampled rounds of more sequences than one 16-row tile of the LM head: the
instances of 32 and 64 rows, and row tiles of 64, whose rows keep their own
place in the random stream and in the per-CTA partials.  Draws, log-sum-exps
and logits against the oracle on the same random streams.
"""
from __future__ import annotations

from dataclasses import replace

import numpy as np
import pytest

import oracle
import synth
from synth.workloads import Workload
from tests.gpu_harness import sample_seqs
from tests.test_gpu_ragged_vocab import TINY_V4000
from tests.test_gpu_sampling import SEED, TAU, compare_sampled, sampled_gpu_round

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,topk", [(17, 1), (40, 3), (64, 8), (65, 1), (130, 8)])
def test_sampled_rows_beyond_one_tile(batch, topk):
    shape = replace(TINY_V4000, name="tiny-v4000-k2", n_steps=2)
    w = Workload("sampled-rows", shape, batch, 8, 40, 2, topk, 71, gain_sigma=0.1)
    W, I = synth.make_weights(w), synth.make_round_inputs(w)
    g = sampled_gpu_round(w, W, I, tau=TAU, seed=SEED, topk=topk)
    assert g["flags"] == 0
    # the last row of each tile and the first of the next among them
    seqs = sorted(set(sample_seqs(batch, 3)) | {b for b in (15, 16, 31, 32, 63, 64, 127, 128) if b < batch})
    o = oracle.draft_round(shape, W, I, topk=topk, want_logits=True, want_hidden=False, seqs=seqs, temperature=TAU,
                           seed=SEED)
    compared, _ = compare_sampled(g, o, seqs, shape.n_steps, TAU)
    assert compared >= len(seqs)
    # the candidate lists are the sorted heads of the logits the round wrote
    order = np.argsort(-g["logits"], axis=2, kind="stable")[..., :topk]
    assert np.array_equal(g["topk_ids"], order)
    assert np.array_equal(g["topk_logits"], np.take_along_axis(g["logits"], order, 2))
