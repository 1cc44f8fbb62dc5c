"""The launch rule of the fused attention (csrc/attn_plan.h, host code without
CUDA), compiled here and asked over batches, KV heads, caches and options."""
from __future__ import annotations

import ctypes
import itertools
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = """
#include "attn_plan.h"
extern "C" void plan(const int *cl, int sms, int ctas, int B, int Hkv, int max_ctx, long long bytes, int warps, int *out) {
    const prism::AttnClusters c{cl[0], {cl[1], cl[2], cl[3], cl[4]}};
    const prism::AttnPlan p = prism::attn_plan(c, {sms, ctas, B, Hkv, max_ctx, bytes}, warps, true);
    out[0] = p.cs;
    out[1] = p.warps;
    out[2] = p.lpt;
}
"""
SMS, RESIDENT = 152, {2: 76, 4: 36, 8: 15, 16: 7}


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2602_01762_gb300", "csrc"),
                    str(d / "shim.cpp"), "-o", so], check=True)
    f = ctypes.CDLL(so).plan

    def call(B, Hkv, max_ctx, *, D=128, es=2, ctas=2, warps=0, resident=RESIDENT):
        most = 16 if resident[16] >= Hkv else 8
        cl, out = (ctypes.c_int * 5)(most, *(resident[c] for c in (2, 4, 8, 16))), (ctypes.c_int * 3)()
        f(cl, SMS, ctas, B, Hkv, max_ctx, ctypes.c_longlong(B * Hkv * max_ctx * D * 2 * es), warps, out)
        return tuple(out)
    return call


def test_clusters_warps_and_order_agree(plan):
    for B, Hkv, ctx, ctas, warps in itertools.product(range(1, 41), (1, 2, 4, 7, 8, 32), (64, 1024, 4096, 32768), (1, 2, 4),
                                                      (0, 4, 8)):
        cs, w, lpt = plan(B, Hkv, ctx, ctas=ctas, warps=warps)
        pairs, small = B * Hkv, B * Hkv * ctx * 512 < 8 << 20
        n = pairs * cs
        where = (B, Hkv, ctx, ctas, warps, cs, w, lpt)
        assert cs in (1, 2, 4, 8, 16) and w in (4, 8), where
        assert cs == 1 or n <= ctas * SMS, where
        # every cluster of four or more is resident at once, sixteen included
        assert small or cs <= 2 or pairs <= RESIDENT[cs], where
        # sixteen only with the kernel they were counted for
        assert cs < 16 or w == 8, where
        assert w == warps if warps else w == 8 or n > SMS, where
        per_wave = SMS * (2 if w == 4 else 1)
        assert lpt == (B > 1 and per_wave < n <= 2 * per_wave), where


def test_an_unknown_residency_limits_nothing(plan):
    unknown = {2: 0, 4: 0, 8: 0, 16: 0}
    assert plan(8, 8, 4096, resident=unknown)[0] == 4             # 64 clusters of 4, up to two CTAs per SM
    assert plan(8, 8, 4096)[0] == 2                               # 36 of them are resident at once


@pytest.mark.parametrize("B,want", [(3, (16, 8)), (4, (8, 8)), (7, (8, 8)), (8, (4, 8))])
def test_two_kv_heads_over_long_caches(plan, B, want):
    """Clusters of sixteen, of which the device holds seven at once, then of eight (fifteen), then of four."""
    assert plan(B, 2, 4096)[:2] == want
