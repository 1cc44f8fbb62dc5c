"""The split-K workspace of a context: every round that the context accepts
finds room for its partial sums, and no more is taken than rounds can use."""
from __future__ import annotations

from dataclasses import replace

import pytest

import synth
from synth.workloads import Workload
from tests.gpu_harness import GpuModel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,width", [(60, 5), (50, 6), (43, 7)])
def test_a_narrower_tree_runs_as_on_a_context_of_its_own_width(batch, width):
    """The gate/up rows of these trees (300 of hidden 256, in three row tiles) are split into more parts than those of
    any width-8 tree of up to 64 sequences.  A context of width 8 launches the same kernels for them as one of the
    tree's own width, whose workspace holds them, and the outputs agree bit for bit."""
    import torch
    from paper_2602_01762_gb300 import Drafter
    from paper_2602_01762_gb300.host import to_device
    shape = replace(synth.workloads.TINY_BF16, name="tiny-k2", n_steps=2)
    w = Workload("narrow-tree", shape, batch, 8, 40, 1, 1, 61, tree_width=width, tree_nodes=6)
    W, I = synth.make_weights(w), synth.make_round_inputs(w)
    model, got = GpuModel(W), []
    try:
        for max_batch, max_width in ((batch, width), (64, 8)):
            dr = Drafter.from_shape(shape, max_batch=max_batch, max_ctx=80, max_new=1, topk=1, max_tree_width=max_width)
            dr.load_shared_weights(model.embed, model.lm_head)
            for k, m in enumerate(W["f_map"]):
                dr.load_step_weights(k, model.modules[m])
            t = {n: to_device(I[n]) for n in ("tokens", "hidden", "n_new", "kv_len")}
            cache = torch.zeros(2, max_batch, shape.n_kv_heads, 80, shape.head_dim, dtype=torch.bfloat16, device="cuda")
            ints = [torch.full((batch, 6), -7, dtype=torch.int32, device="cuda") for _ in range(3)]
            scores = torch.zeros(batch, 6, device="cuda")
            rows = torch.zeros(2, batch, width, shape.vocab, device="cuda")
            for _ in range(2):
                dr.draft_tree(t["tokens"], t["hidden"], t["n_new"], t["kv_len"], cache[0], cache[1], width, *ints, scores,
                              row_logits=rows)
            assert dr.sync_status() == 0
            got.append((dr.round_launches(), *ints, scores, rows))
            dr.close()
    finally:
        model.close()
    assert got[0][0] == got[1][0]
    assert all(torch.equal(a, b) for a, b in zip(got[0][1:], got[1][1:]))


def test_a_prompts_rows_take_no_room_in_the_mlp():
    """Only the fusion and QKV multiply every row of step 1.  At 64 sequences of the Llama-3-8B shape with 6 tokens each
    the largest split is QKV's, three slices of 384 rows; gate/up, which runs on 64 rows, would need 84 MB for 384."""
    import torch
    from paper_2602_01762_gb300 import Drafter
    s = synth.workloads.L3_8B
    qkv = (s.n_q_heads + 2 * s.n_kv_heads) * s.head_dim

    def taken(max_new):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        dr = Drafter.from_shape(s, max_batch=64, max_ctx=128, max_new=max_new, topk=1)
        used = before - torch.cuda.mem_get_info()[0]
        dr.close()
        return used
    taken(1)                                                    # loads the kernels
    own = 5 * 64 * (s.hidden * 4 + qkv * 4 + 2 * s.hidden * 2)  # x0, QKV and the bf16 fusion rows of 5 tokens more
    slices = 3 * 384 * qkv * 4
    assert taken(6) - taken(1) <= own + slices + (4 << 20)      # and the allocator's 2 MB steps
