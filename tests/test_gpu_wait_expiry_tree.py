"""Bounded waits that give up in a tree round: the tree's attention kernel, of
one and of several stages and CTAs, and the projections of its rows report the
timeout and wind down, and the next round of the same context is bit for bit
the round before.  (The chain's kernels: test_gpu_wait_expiry.)
"""
from __future__ import annotations

import pytest

import synth
from synth.workloads import Workload
from tests.gpu_harness import GpuModel
from tests.test_gpu_ragged_vocab import TINY_V4000
from tests.test_gpu_wait_expiry import PRISM_ERR_TIMEOUT, TIMEOUT_BIT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,width,ctx", [(1, 4, 3000), (3, 8, 40)])
def test_tree_waits_that_give_up_report_timeout_and_the_context_recovers(batch, width, ctx):
    import torch
    from paper_2602_01762_gb300 import Drafter
    from paper_2602_01762_gb300.host import to_device
    w = Workload("tree-expiry", TINY_V4000, batch, ctx, ctx, 2, 1, 81, gain_sigma=0.1, tree_width=width, tree_nodes=9)
    W, I = synth.make_weights(w), synth.make_round_inputs(w)
    model = GpuModel(W)
    dr = Drafter.from_shape(w.shape, max_batch=batch, max_ctx=int(I["max_ctx"]), max_new=2, topk=1, max_tree_width=width)

    def tree(polls):
        dr.set_option("wait_polls", polls)
        t = {n: to_device(I[n]) for n in ("tokens", "hidden", "n_new", "kv_len", "k_cache", "v_cache")}
        ints = [torch.full((batch, 9), -7, dtype=torch.int32, device="cuda") for _ in range(3)]
        out = ints + [torch.zeros(batch, 9, device="cuda"),
                      torch.zeros(w.shape.n_steps, batch, width, w.shape.vocab, device="cuda")]
        dr.draft_tree(t["tokens"], t["hidden"], t["n_new"], t["kv_len"], t["k_cache"], t["v_cache"], width, *out[:4],
                      row_logits=out[4])
        return dr.sync_status(), out + [t["k_cache"], t["v_cache"]]
    try:
        dr.load_shared_weights(model.embed, model.lm_head)
        for k, m in enumerate(W["f_map"]):
            dr.load_step_weights(k, model.modules[m])
        flags, want = tree(0)
        assert flags == 0 and dr.last_status == 0
        flags, _ = tree(-1)
        assert flags & TIMEOUT_BIT and dr.last_status == PRISM_ERR_TIMEOUT
        tree(1)
        assert dr.last_status in (0, PRISM_ERR_TIMEOUT)
        flags, got = tree(0)
        assert flags == 0 and dr.last_status == 0
        assert all(torch.equal(a, b) for a, b in zip(want, got))
    finally:
        dr.close()
        model.close()
