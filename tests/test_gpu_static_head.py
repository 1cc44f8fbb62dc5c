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


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("rows,hidden,topk", [(1, 256, 1), (16, 256, 1), (17, 256, 1), (3, 256, 8), (64, 256, 5), (41, 8192, 8)])
def test_places_without_a_candidate(dtype, rows, hidden, topk):
    """NaN logits are no candidates, and a place left over holds id 0x7FFFFFFF and logit -inf, whatever the type and
    the route: the packed top-1, lists in one pass and in several.  Here three tokens of nine have a number, of which
    one is -inf in the odd rows; in the last row none has."""
    import torch
    from paper_2602_01762_gb300 import lm_head_topk_static
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    lm = torch.full((9, hidden), float("nan"), device="cuda", dtype=dt)
    lm[2], lm[5], lm[8] = 0.5, 0.25, 0.0
    lm[8, 1] = float("-inf")
    h = torch.ones(rows, hidden, device="cuda")
    h[::2, 1] = 0.0                          # -inf * 0: NaN
    h[-1] = float("nan")
    i32 = dict(dtype=torch.int32, device="cuda")
    draft, ids, flags = torch.full((rows,), -7, **i32), torch.full((rows, topk), -7, **i32), torch.full((1,), -7, **i32)
    top = torch.zeros(rows, topk, device="cuda")
    lm_head_topk_static(h, None, lm, draft, ids, top, None, flags)
    assert int(flags) == 0
    none, inf = 0x7FFFFFFF, float("inf")
    for r in range(rows):
        n = sum(h[r].tolist()) if r < rows - 1 else 0
        found = [] if r == rows - 1 else [(2, 0.5 * n), (5, 0.25 * n)] + ([(8, -inf)] if r % 2 else [])
        want = (found + [(none, -inf)] * topk)[:topk]
        assert ids[r].tolist() == [i for i, _ in want] and top[r].tolist() == [v for _, v in want], r
        assert int(draft[r]) == want[0][0]
