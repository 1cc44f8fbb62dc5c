"""The fp32 projection kernel where its plan divides: 1, 2, 4 or 8 activation
rows per warp, 1 to 4 row groups per pass, several passes, contractions shared
by 1 to 8 warps or not a multiple of a warp's step, items that reach past the
last unit, more CTAs than items, and selections in several chunks.
"""
from __future__ import annotations

import pytest

import synth
from synth.workloads import Shape, Workload
from tests.gpu_harness import sample_seqs
from tests.test_gpu_round import _check
from tests.test_gpu_tree import ragged

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,hidden,vocab,topk,norm", [
    (1, 8, 8, 8, True), (1, 1024, 9001, 1, True), (2, 136, 601, 3, False), (3, 1024, 32000, 4, True),
    (5, 4096, 5003, 8, True), (9, 1032, 4000, 8, True), (17, 1024, 40001, 2, True), (33, 512, 41000, 8, False),
    (64, 4096, 9000, 1, True)])
def test_f32_head(rows, hidden, vocab, topk, norm):
    import torch
    from paper_2602_01762_gb300 import lm_head_topk_static
    g = torch.Generator(device="cuda").manual_seed(rows * 31 + topk)
    lm = torch.randn(vocab, hidden, generator=g, device="cuda") / hidden ** 0.5
    h = torch.randn(rows, hidden, generator=g, device="cuda") * 2
    gain = 1 + 0.1 * torch.randn(hidden, generator=g, device="cuda") if norm else None
    lm[3, 1] = float("nan")                  # its logits are no candidates
    i32 = dict(dtype=torch.int32, device="cuda")
    draft, ids, flags = torch.full((rows,), -1, **i32), torch.full((rows, topk), -1, **i32), torch.full((1,), -1, **i32)
    top, logits = torch.zeros(rows, topk, device="cuda"), torch.zeros(rows, vocab, device="cuda")
    x = h.double()
    if norm:
        x = x * torch.rsqrt(x.square().mean(1, keepdim=True) + 1e-5) * gain.double()
    want = x @ lm.double().T
    lm_head_topk_static(h, gain, lm, draft, ids, top, logits, flags)
    assert int(flags) == 0
    keep = [u for u in range(vocab) if u != 3]
    # a lane's sum takes hidden / 64 roundings, the lanes' and segments' 16, the norm's row 4 more per element; partial
    # sums stay below 12 (rows of variance at most 4, unit-variance weights over hidden^1/2)
    err = (logits.double() - want)[:, keep].abs().max().item()
    assert err <= 2.0 ** -24 * (hidden / 64 + 20) * 12, err
    assert bool(logits[:, 3].isnan().all())
    z = logits.clone()
    z[:, 3] = float("-inf")
    own = torch.sort(z, dim=1, descending=True, stable=True)
    n = min(topk, vocab - 1)
    assert torch.equal(ids.long()[:, :n], own.indices[:, :n]) and torch.equal(top[:, :n], own.values[:, :n])
    assert torch.equal(draft.long(), own.indices[:, 0])
    if topk > n:                             # fewer candidates than places
        assert bool((ids[:, n:] == 0x7FFFFFFF).all()) and bool((top[:, n:] == float("-inf")).all())


@pytest.mark.parametrize("batch,n_new,topk", [(1, 1, 1), (3, 5, 4), (9, 2, 8), (24, 5, 3)])
def test_f32_round(batch, n_new, topk):
    shape = Shape("f32-odd", 520, 5, 1, 64, 1000, 2003, 3, "f32", 10000.0)
    w = Workload("f32-odd", shape, batch, 8, 40, n_new, topk, 21, gain_sigma=0.1)
    W, I = synth.make_weights(w), synth.make_round_inputs(w)
    _, _, rep = _check(w, W, ragged(w, I) if n_new > 1 else I, sample_seqs(batch, 3), topk=topk)
    assert rep["ids_compared"] >= 1
