"""The LM head that allocates nothing, where its route divides: one 16-row
tile with the packed top-1, more rows or candidates through the top-8 lists,
row tiles, and rows that need several passes because the static array holds
only part of them beside the lists.  Checked against the same rows in 64 bits.
"""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,hidden,vocab,topk,norm", [
    (1, 256, 4000, 1, True), (16, 256, 4096, 1, True), (17, 256, 4000, 1, False), (16, 1024, 9001, 8, True),
    (33, 1016, 4000, 3, True), (40, 8192, 9000, 8, True), (41, 8192, 9000, 2, False), (64, 8192, 1000, 1, True),
    (64, 24, 8, 8, True)])
def test_static_head_routes(rows, hidden, vocab, topk, norm):
    import torch
    from paper_2602_01762_gb300 import lm_head_topk_static
    g = torch.Generator(device="cuda").manual_seed(rows * 31 + topk)
    lm = (torch.randn(vocab, hidden, generator=g, device="cuda") / hidden ** 0.5).bfloat16()
    h = torch.randn(rows, hidden, generator=g, device="cuda") * 2
    gain = (1 + 0.1 * torch.randn(hidden, generator=g, device="cuda")).bfloat16() if norm else None
    i32 = dict(dtype=torch.int32, device="cuda")
    draft, ids, flags = torch.full((rows,), -1, **i32), torch.full((rows, topk), -1, **i32), torch.full((1,), -1, **i32)
    top, logits = torch.zeros(rows, topk, device="cuda"), torch.zeros(rows, vocab, device="cuda")
    x = h * torch.rsqrt(h.double().square().mean(1, keepdim=True) + 1e-5).float() * gain.float() if norm else h
    want = x.bfloat16().double() @ lm.double().T
    for _ in range(2):                      # the second call finds the scratch as the first left it
        lm_head_topk_static(h, gain, lm, draft, ids, top, logits, flags)
        assert int(flags) == 0
        # fp32 sums of `hidden` products of unit-variance rows, and one bf16 rounding that a last bit of the norm may
        # flip (2^-8 of one element, of weight hidden^-1/2)
        err = (logits.double() - want).abs().max().item()
        assert err <= 2 ** -8 * 12 / hidden ** 0.5 + 1e-5, err
        own = torch.sort(logits, dim=1, descending=True, stable=True)
        assert torch.equal(ids.long(), own.indices[:, :topk]) and torch.equal(top, own.values[:, :topk])
        assert torch.equal(draft.long(), own.indices[:, 0])
