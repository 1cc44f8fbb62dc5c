"""A tree round whose logits hold a NaN: every row's log-sum-exp and so every
score is NaN.  Such scores rank as -inf, in pool order, so the verified tree
has exactly n_nodes entries and nothing is written behind its outputs."""
from __future__ import annotations

import pytest

import oracle
import synth
from synth.workloads import Workload
from tests.gpu_harness import GpuModel
from tests.test_gpu_ragged_vocab import TINY_V4000

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,width,n_nodes", [(1, 4, 5), (3, 2, 3)])
def test_nan_scores_rank_last_in_pool_order(batch, width, n_nodes):
    import torch
    from paper_2602_01762_gb300 import Drafter
    from paper_2602_01762_gb300.host import to_device
    w = Workload("tree-nan", TINY_V4000, batch, 8, 40, 1, 1, 51, tree_width=width, tree_nodes=n_nodes)
    W, I = dict(synth.make_weights(w)), synth.make_round_inputs(w)
    W["lm_head"] = W["lm_head"].copy()
    W["lm_head"][7] = 0x7FC0
    model = GpuModel(W)
    K, P = w.shape.n_steps, oracle.pool_size(w.shape.n_steps, width)
    dr = Drafter.from_shape(w.shape, max_batch=batch, max_ctx=int(I["max_ctx"]), max_new=1, topk=1, max_tree_width=width)
    try:
        dr.load_shared_weights(model.embed, model.lm_head)
        for k, m in enumerate(W["f_map"]):
            dr.load_step_weights(k, model.modules[m])
        t = {n: to_device(I[n]) for n in ("tokens", "hidden", "n_new", "kv_len", "k_cache", "v_cache")}

        def guarded(n, dtype):          # n entries per sequence, and room behind them that no one may write
            room = torch.full((batch * n + batch * P + 64,), -7, dtype=dtype, device="cuda")
            return room, room[:batch * n].view(batch, n)
        rooms, outs = zip(*[guarded(n_nodes, dt) for dt in (torch.int32,) * 3 + (torch.float32,)])
        pool = torch.full((batch, P), -7, dtype=torch.int32, device="cuda")
        front = torch.full((batch, K, width), -7, dtype=torch.int32, device="cuda")
        dr.draft_tree(t["tokens"], t["hidden"], t["n_new"], t["kv_len"], t["k_cache"], t["v_cache"], width, *outs,
                      pool_tokens=pool, frontier=front)
        assert dr.sync_status() == 0
    finally:
        dr.close()
        model.close()
    for room in rooms:
        assert bool((room[batch * n_nodes:] == -7).all())
    assert bool(outs[3].isnan().all())
    assert torch.equal(outs[0], pool[:, :n_nodes]) and bool((pool >= 0).all()) and bool((pool != 7).all())
    starts = torch.tensor([0] + [width + (k - 2) * width * width for k in range(2, K + 1)], device="cuda")
    assert torch.equal(front.long(), (starts[:, None] + torch.arange(width, device="cuda"))[None].expand(batch, -1, -1))
