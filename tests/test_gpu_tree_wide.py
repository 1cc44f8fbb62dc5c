"""Tree attention of more than 16 row-head pairs keeps fp32 queries, held as
three bf16 parts."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from oracle import to_bf16_bits as f32_to_bf16
from synth.workloads import Shape, Workload
from tests.parity import rel_l2
from tests.test_gpu_tree import gpu_tree

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [5, 8])
def test_queries_keep_all_their_bits(width):
    """Scores that are sums of large terms which cancel: q holds m_a z and m_b z (z of some 20 bits), the keys
    +-2^13 m_b and -+2^13 m_a, and the rotary angles of these dims are below 2^-15, so that every score is 0 and
    attention an even mean.  The terms reach 2^19 and 24 of them are added: fp32 sums leave less than 0.1 of a
    score, a query of two bf16 parts (16 bits) 1.2."""
    shape = Shape("tree-bits", 256, 4, 1, 64, 512, 4000, 2, "bf16", 1e30)
    w = Workload("tree-bits", shape, 1, 400, 400, 1, 1, 91, tree_width=width, tree_nodes=6)
    W, I = synth.make_weights(w), synth.make_round_inputs(w)
    rng = np.random.default_rng(91)
    ratios = [(3, 5), (5, 7), (7, 9), (9, 11), (11, 13), (3, 7), (5, 9), (7, 11), (9, 13), (3, 11), (5, 13), (7, 13)]
    for mod in W["modules"].values():
        mod["w_qkv"] = mod["w_qkv"].copy()
        mod["w_qkv"][:5 * 64] = 0                        # queries and new keys
        mod["w_o"] = f32_to_bf16(synth.bf16_to_f32(mod["w_o"]) * 8)
    qw = np.zeros((4, 64, 256), np.float32)
    keys = np.zeros(I["k_cache"].shape, np.float32)
    for p, (ma, mb) in enumerate(ratios):
        a = 8 + 2 * p
        for h in range(4):
            c1, c2 = rng.choice(256, 2, replace=False)
            z1, z2 = rng.integers(8, 16, 2) / 8 * [1, 2 ** -6]
            for dim, m in ((a, ma), (a + 1, mb)):
                qw[h, dim, c1], qw[h, dim, c2] = m * z1, m * z2
        sign = rng.choice([-1.0, 1.0], 400)
        keys[0, 0, :400, a], keys[0, 0, :400, a + 1] = sign * mb * 2 ** 13, -sign * ma * 2 ** 13
    assert np.array_equal(synth.bf16_to_f32(f32_to_bf16(qw)), qw) and np.array_equal(synth.bf16_to_f32(f32_to_bf16(keys)), keys)
    W["modules"][1]["w_qkv"][:256] = f32_to_bf16(qw).reshape(256, 256)
    I["k_cache"] = f32_to_bf16(keys)
    I["v_cache"] = f32_to_bf16(synth.bf16_to_f32(I["v_cache"]) * 8)
    g = gpu_tree(w, W, I, width=width, n_nodes=6)
    assert g["flags"] == 0
    o = oracle.draft_tree(shape, W, I, width=width, n_nodes=6, seqs=[0],
                          follow={"pool_tokens": g["pool_tokens"], "frontier": g["frontier"]})
    assert rel_l2(g["row_logits"][0, 0, 0], o["row_logits"][0, 0, 0]) < 0.01
    for j in range(width):
        assert rel_l2(g["row_logits"][0, 1, j], o["row_logits"][0, 1, j]) < 0.1, j
