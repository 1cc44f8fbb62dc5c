"""Gate/up of one bf16 row (four weight rows per warp): a contraction that is
not a multiple of a warp's step, CTAs of uneven numbers of items, layers on either
side of the size below which the ring kernel keeps them.
"""
from __future__ import annotations

import pytest

import synth
from synth.workloads import Shape, Workload
from tests.test_gpu_round import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,ffn", [(520, 1000), (1032, 30008), (2056, 16104), (4096, 7800)])
def test_one_row_gate_up(hidden, ffn):
    shape = Shape("gate-up-row", hidden, 4, 1, 64, ffn, 2000, 3, "bf16", 10000.0)
    w = Workload("gate-up-row", shape, 1, 20, 40, 1, 2, 41, gain_sigma=0.1)
    W, I = synth.make_weights(w), synth.make_round_inputs(w)
    _, _, rep = _check(w, W, I, [0], topk=2)
    assert rep["ids_compared"] >= 1
