// How the fused attention is launched (host only, no CUDA): CTAs per cluster,
// compute warps per CTA and the order of the sequences.
#pragma once

namespace prism {

// Cluster sizes of the fused attention on this device: the largest (16 only where
// the clusters of one sequence can be resident at once, else 8), and how many
// clusters of 2, 4, 8 and 16 CTAs can be resident at once (0: unknown).  On a
// GB300, of the 8-warp kernel: 76, 36, 15 and 7.
struct AttnClusters {
    int most, resident[4];
};

struct AttnSizes {
    int sms, ctas_per_sm;   // SMs; option attn_ctas_per_sm
    int B, Hkv, max_ctx;
    long long cache_bytes;  // of the K and V rows of B sequences at full capacity
};

struct AttnPlan {
    int cs, warps, lpt;     // lpt: the longest sequences first
};

// Bytes of K and V below which clusters and warps keep the choice below, and
// cache rows beyond which two-CTA clusters keep 8 warps.  Both look at the cache's
// capacity: the contexts are device data that the host does not know at a launch.
constexpr long long kAttnSmallCache = 8LL << 20;
constexpr int kAttnLongCtx = 3072;   // see attn_plan

inline bool attn_small_cache(const AttnSizes &z) { return z.cache_bytes < kAttnSmallCache; }

// CTAs per (sequence, KV head): halved while they exceed ctas_per_sm per SM, and
// while the device cannot hold all clusters at once: the second wave of clusters of
// 4 or more starts only when that many SMs of one GPC are free, and costs a whole
// launch's latency again (8B shape, batch 4, contexts to 4096, clusters of 8 and of 4: 1405
// us a round and 1325; the 7B shape at batch 1 1069 and 980; the tree of 4 sequences
// 1192 and 1116; hidden 1024 with 2 KV heads, batch 4, contexts to 8000, clusters of
// 16 and of 8: 280 and 261).  pair_fits: clusters of two may take two waves.  Small
// caches keep their clusters: the order of their sums decides nearly tied
// candidates of small drafters (tiny drafter, batch 8, contexts to 200: 147 us, 177 so).
inline int attn_cluster(const AttnClusters &cl, const AttnSizes &z, int most, bool pair_fits) {
    const long long pairs = (long long)z.B * z.Hkv;
    auto fits = [&](int cs) {
        const int n = cl.resident[cs == 16 ? 3 : cs == 8 ? 2 : cs == 4 ? 1 : 0];
        return attn_small_cache(z) || (cs == 2 && pair_fits) || n == 0 || pairs <= n;
    };
    int cs = most;
    while (cs > 1 && (pairs * cs > (long long)z.ctas_per_sm * z.sms || !fits(cs))) cs /= 2;
    return cs;
}

// The chain's attention.  want_warps: option attn_warps (0: by rule); want_lpt: option attn_lpt.
inline AttnPlan attn_plan(const AttnClusters &cl, const AttnSizes &z, int want_warps, bool want_lpt) {
    AttnPlan p;
    // clusters of 16 are checked for the 8-warp kernel only
    p.cs = attn_cluster(cl, z, want_warps == 4 && cl.most > 8 ? 8 : cl.most, true);
    // more CTAs than SMs: 4-warp CTAs, two per SM, so that one streams while
    // the other starts or merges (8B shape, top-8, contexts 512 to 4096, batch
    // 64: 2050 us a round with 8 warps, 2009 with 4; 7B shape, batch 16, 1937
    // and 1875).  Clusters of two in two waves over long caches keep 8 warps:
    // twice the bytes in flight per CTA and, with the longest sequences first,
    // a short tail where the contexts are uneven.  8B shape, 3 steps, batch 10 / 16, us
    // a round with 8 warps and with 4: contexts 512 to 2048 822 / 885 and 818 / 869, to
    // 3040 824 / 892 and 831 / 888, to 4096 846 / 902 and 850 / 906, to 8000 863 / 955 and
    // 909 / 982 (7B shape, batch 3, 535 and 568).  Even contexts would take 4 warps at any
    // length (4096: 912 / 960 and 861 / 938), and so would short ones in a long cache
    // (512 to 2048 of 16384: 819 / 885 and 820 / 870), which a launch cannot tell.
    // Small caches: one wave of single CTAs only (as for their clusters)
    const long long n_ctas = (long long)z.B * z.Hkv * p.cs;
    const bool long_pairs = p.cs == 2 && z.B > 1 && z.max_ctx > kAttnLongCtx;
    const bool four = p.cs <= 8 && (attn_small_cache(z) ? p.cs == 1 && n_ctas <= 2LL * z.sms : !long_pairs);
    p.warps = want_warps ? want_warps : n_ctas > z.sms && four ? 4 : 8;
    // more than one wave of CTAs but at most two: the longest sequences
    // first (with more waves the hardware's scheduling already evens
    // them out and each CTA's ranking of the sequences costs more than
    // the order gains; 8B shape, batch 64, contexts 512 to 4096: 2009 us
    // with the order, 2090 without; batch 24, one wave: 1644 and 1630)
    const long long per_wave = (long long)z.sms * (p.warps == 4 ? 2 : 1);
    p.lpt = want_lpt && z.B > 1 && z.B <= 256 && n_ctas > per_wave && n_ctas <= 2 * per_wave;
    return p;
}

}  // namespace prism
