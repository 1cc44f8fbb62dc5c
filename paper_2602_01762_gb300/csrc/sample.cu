// Sampled drafting and speculative-sampling acceptance (Sec. 2 at a
// temperature T > 0), sm_103a.
//
// Drafting: each draft token is drawn from p_draft = softmax(z / T) by the Gumbel-max rule: the
// argmax of z_i / T + G_i with G_i = -log(-log U_i) is distributed as
// softmax(z / T).  The logits of one row are split over many CTAs; each keeps
// a running (max, sum of exp) of z / T and its best perturbed score, and the
// last CTA of the row merges them in CTA order and writes the token and
// lse = log sum_i exp(z_i / T), so that p_draft(x) = exp(z_x / T - lse).  A
// streamed tcgen05 LM head draws in its own epilogue (gemv_tc.cu); sample_kernel
// here reads the logits back after any other LM head.
//
// Acceptance: one cluster per sequence tests the K drafted positions; x is
// accepted when r * p_draft(x) < p_target(x) (r < min(1, p_target /
// p_draft)); the first rejected position draws its replacement from
// max(0, p_target - p_draft) by an inverse-CDF search over the vocabulary (a
// residual that is zero everywhere falls back to p_target); after a full
// accept the extra token is drawn from p_target at position K.
//
// Random numbers: the n-th output of SplitMix64 (Steele, Lea and Flood,
// OOPSLA 2014) started from state `seed`, with the counter
// n = (stream << 60) | (b << 40) | (k << 32) | i, mapped to (0, 1) as
// ((x >> 41) + 1/2) / 2^23 (exact in float32).  Streams: 1 draft sampling
// (i = token id), 2 the acceptance test of position k, 3 the token drawn at
// position k (k = K: the extra token after a full accept).
#include "common.cuh"

namespace prism {

namespace {

constexpr int kSampleThreads = 256;

// (max, sum of exp(v - max)) of two parts, combined.
__device__ __forceinline__ void lse_merge(float &m, float &s, float m2, float s2) {
    if (m2 == -INFINITY) return;
    if (m == -INFINITY) { m = m2; s = s2; return; }
    if (m2 > m) { s = s * expf(m - m2) + s2; m = m2; }
    else s += s2 * expf(m2 - m);
}

// grid (blocks per row, B); a CTA takes `chunk` consecutive logits of row b.
__global__ void __launch_bounds__(kSampleThreads) sample_kernel(const SampleArgs a) {
    __shared__ float s_m[kSampleThreads / 32], s_s[kSampleThreads / 32], s_v[kSampleThreads / 32];
    __shared__ int s_i[kSampleThreads / 32];
    __shared__ int s_last;
    pdl_trigger();
    pdl_wait();
    const int b = blockIdx.y, blk = blockIdx.x, nblk = gridDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t seed = *a.seed;
    const float inv_t = 1.0f / a.temperature;
    const float *z = a.logits + ((size_t)b * a.K + a.step - 1) * a.V;
    const int lo = blk * a.chunk, hi = min(a.V, lo + a.chunk);
    float m = -INFINITY, s = 0.f, bv = -INFINITY;
    int bi = 0x7FFFFFFF;
    for (int i = lo + tid; i < hi; i += kSampleThreads) {
        const float v = z[i] * inv_t;
        lse_merge(m, s, v, 1.f);
        const float u = uniform01(seed, 1, (uint32_t)b, (uint32_t)(a.step - 1), (uint32_t)i);
        const float g = v - logf(-logf(u));
        if (better(g, i, bv, bi)) { bv = g; bi = i; }
    }
    // block: warps in a fixed tree, then warp 0 over the warps in order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float m2 = __shfl_xor_sync(0xFFFFFFFFu, m, o), s2 = __shfl_xor_sync(0xFFFFFFFFu, s, o);
        const float v2 = __shfl_xor_sync(0xFFFFFFFFu, bv, o);
        const int i2 = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
        lse_merge(m, s, m2, s2);
        if (better(v2, i2, bv, bi)) { bv = v2; bi = i2; }
    }
    if (lane == 0) { s_m[warp] = m; s_s[warp] = s; s_v[warp] = bv; s_i[warp] = bi; }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < kSampleThreads / 32; ++w) {
            lse_merge(m, s, s_m[w], s_s[w]);
            if (better(s_v[w], s_i[w], bv, bi)) { bv = s_v[w]; bi = s_i[w]; }
        }
        float *part = a.part + ((size_t)b * a.max_blocks + blk) * 4;
        part[0] = m;
        part[1] = s;
        part[2] = bv;
        part[3] = __int_as_float(bi);
        __threadfence();
        s_last = atomicAdd(a.counter + b, 1) == nblk - 1;
    }
    __syncthreads();
    if (!s_last || warp != 0) return;
    // the row's last CTA: lane l merges partials l, l + 32, ... (loads first),
    // then the lanes merge in a fixed butterfly order
    __threadfence();
    constexpr int kPer = kSampleMaxBlocks / 32;
    float pm[kPer], ps[kPer], pv[kPer];
    int pi[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int q = lane + 32 * i;
        const float4 v = q < nblk ? __ldcg((const float4 *)(a.part + ((size_t)b * a.max_blocks + q) * 4))
                                  : make_float4(-INFINITY, 0.f, -INFINITY, __int_as_float(0x7FFFFFFF));
        pm[i] = v.x;
        ps[i] = v.y;
        pv[i] = v.z;
        pi[i] = __float_as_int(v.w);
    }
    float M = -INFINITY, S = 0.f, BV = -INFINITY;
    int BI = 0x7FFFFFFF;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        lse_merge(M, S, pm[i], ps[i]);
        if (better(pv[i], pi[i], BV, BI)) { BV = pv[i]; BI = pi[i]; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float m2 = __shfl_xor_sync(0xFFFFFFFFu, M, o), s2 = __shfl_xor_sync(0xFFFFFFFFu, S, o);
        const float v2 = __shfl_xor_sync(0xFFFFFFFFu, BV, o);
        const int i2 = __shfl_xor_sync(0xFFFFFFFFu, BI, o);
        lse_merge(M, S, m2, s2);
        if (better(v2, i2, BV, BI)) { BV = v2; BI = i2; }
    }
    if (lane == 0) {
        const size_t o = (size_t)b * a.K + a.step - 1;
        a.draft[o] = BI;
        a.lse[o] = M + logf(S);
        a.counter[b] = 0;
    }
}

// Inverse-CDF draw over the vocabulary by a cluster of kAccCtas CTAs.  The V
// weights are cut into groups of 128 m consecutive tokens (m so that a CTA has
// at most kAccGroups groups) and the groups into one contiguous range per CTA.
// Each warp sums its groups with coalesced loads, several groups' loads in
// flight; a scan of the CTA's group sums and the CTAs' totals, read through
// distributed shared memory, gives every group its bounds on the cumulative
// sum, and the one CTA whose range holds u * total searches the one group that
// does, a warp at a time.  It is a chain of latencies on a few SMs: one CTA of
// 1024 threads per sequence, each thread walking its own 126 tokens (128-byte
// strides between neighbouring lanes, both rows through one SM), took
// 64 us for 8 sequences of 128256 tokens; the cluster takes 13 us.
constexpr int kAccCtas = 8;
constexpr int kAccThreads = 512;
constexpr int kAccWarps = kAccThreads / 32;
constexpr int kAccGroups = 512;

struct AccShared {
    float gsum[kAccGroups];     // group sums, then their inclusive scan
    float total;                // the CTA's sum
    float wlast[kAccWarps];
    float last;                 // last token of the CTA with a positive weight, -1: none (as a float's bits)
    float tok;                  // the drawn token in the CTA that owns it, else -1 (as a float's bits)
};

// Returns the token in every thread of the cluster, or -1 when every weight is 0.
template <typename W>
__device__ int draw_cluster(W w, int V, float u, AccShared &sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, r = blockIdx.x % kAccCtas;
    int gs = 128;
    while (((V + gs - 1) / gs + kAccCtas - 1) / kAccCtas > kAccGroups) gs *= 2;
    const int ngroups = (V + gs - 1) / gs;
    const int g0 = (int)((long)r * ngroups / kAccCtas), ng = (int)((long)(r + 1) * ngroups / kAccCtas) - g0;
    int last = -1;
    for (int g = warp; g < ng; g += 2 * kAccWarps) {
        float v[2][4] = {};
        float sum[2] = {0.f, 0.f};
        for (int o = 0; o < gs; o += 128) {
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int gg = g + q * kAccWarps, i = (g0 + gg) * gs + o + 32 * j + lane;
                    v[q][j] = gg < ng && i < V ? w(i) : 0.f;
                    if (v[q][j] > 0.f) last = max(last, i);
                }
#pragma unroll
            for (int q = 0; q < 2; ++q) sum[q] += (v[q][0] + v[q][1]) + (v[q][2] + v[q][3]);
        }
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) {
            sum[0] += __shfl_xor_sync(0xFFFFFFFFu, sum[0], s);
            sum[1] += __shfl_xor_sync(0xFFFFFFFFu, sum[1], s);
        }
        if (lane == 0) {
            sh.gsum[g] = sum[0];
            if (g + kAccWarps < ng) sh.gsum[g + kAccWarps] = sum[1];
        }
    }
    last = __reduce_max_sync(0xFFFFFFFFu, last);
    if (lane == 0) sh.wlast[warp] = __int_as_float(last);
    if (tid == 0) sh.tok = __int_as_float(-1);
    __syncthreads();
    if (warp == 0) {
        float base = 0.f;
        for (int g = 0; g < ng; g += 32) {
            float c = g + lane < ng ? sh.gsum[g + lane] : 0.f;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const float x = __shfl_up_sync(0xFFFFFFFFu, c, s);
                if (lane >= s) c += x;
            }
            if (g + lane < ng) sh.gsum[g + lane] = base + c;
            base += __shfl_sync(0xFFFFFFFFu, c, 31);
        }
        const int l = __reduce_max_sync(0xFFFFFFFFu, lane < kAccWarps ? __float_as_int(sh.wlast[lane]) : -1);
        if (lane == 0) {
            sh.total = ng > 0 ? sh.gsum[ng - 1] : 0.f;
            sh.last = __int_as_float(l);
        }
    }
    cluster_sync_all();
    // CTA q covers [pre(q), pre(q) + total(q)), summed alike in every CTA
    float total = 0.f, pre = 0.f;
    int all_last = -1;
#pragma unroll
    for (int q = 0; q < kAccCtas; ++q) {
        if (q == r) pre = total;
        total += dsmem_ld(&sh.total, (uint32_t)q);
        all_last = max(all_last, __float_as_int(dsmem_ld(&sh.last, (uint32_t)q)));
    }
    const float target = u * total, own = sh.total;
    if (warp == 0 && own > 0.f && pre <= target && target < pre + own) {
        // the first group whose end lies beyond the target (the last one's does)
        int g = 0;
        for (; g < ng; g += 32) {
            const unsigned m = __ballot_sync(0xFFFFFFFFu, g + lane < ng && pre + sh.gsum[g + lane] > target);
            if (m) { g += __ffs(m) - 1; break; }
        }
        g = min(g, ng - 1);
        float c = g > 0 ? pre + sh.gsum[g - 1] : pre;
        int tok = -1, seen = -1;
        for (int o = 0; o < gs && tok < 0; o += 32) {
            const int i = (g0 + g) * gs + o + lane;
            const float wi = i < V ? w(i) : 0.f;
            float in = wi;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const float x = __shfl_up_sync(0xFFFFFFFFu, in, s);
                if (lane >= s) in += x;
            }
            const unsigned m = __ballot_sync(0xFFFFFFFFu, wi > 0.f && c + in > target);
            const unsigned pos = __ballot_sync(0xFFFFFFFFu, wi > 0.f);
            if (m) tok = (g0 + g) * gs + o + __ffs(m) - 1;
            if (pos) seen = (g0 + g) * gs + o + 31 - __clz(pos);
            c += __shfl_sync(0xFFFFFFFFu, in, 31);
        }
        // the bounds came from sums in another order: the group's last positive weight
        if (lane == 0) sh.tok = __int_as_float(tok >= 0 ? tok : seen);
    }
    cluster_sync_all();
    int tok = -1;
#pragma unroll
    for (int q = 0; q < kAccCtas; ++q) tok = max(tok, __float_as_int(dsmem_ld(&sh.tok, (uint32_t)q)));
    // u * total rounded onto the top of the range: the last positive weight
    if (tok < 0 && total > 0.f) tok = all_last;
    cluster_sync_all();         // every CTA has read before a second draw (or an exit) ends the values' life
    return tok;
}

// One cluster per sequence.  Every CTA makes the K acceptance tests at once
// (one lane each; K <= 16) and so finds the same first rejection.
__global__ void __launch_bounds__(kAccThreads) accept_sampled_kernel(const AcceptSampledArgs a) {
    __shared__ AccShared sh;
    __shared__ int s_acc;
    const int b = blockIdx.x / kAccCtas, rank = blockIdx.x % kAccCtas, tid = threadIdx.x, K = a.K, V = a.V;
    const uint64_t seed = *a.seed;
    const float inv_t = 1.0f / a.temperature;
    if (tid < 32) {
        bool reject = false, bad = false;
        if (tid < K) {
            const size_t row = (size_t)b * K + tid;
            int x = a.draft[row];
            bad = x < 0 || x >= V;
            if (bad) x = 0;
            const float pd = expf(a.logits[row * V + x] * inv_t - a.lse[row]);
            const float r = uniform01(seed, 2, (uint32_t)b, (uint32_t)tid, 0);
            reject = !(r * pd < a.target[((size_t)b * (K + 1) + tid) * V + x]);
        }
        const unsigned rej = __ballot_sync(0xFFFFFFFFu, reject);
        const int acc = rej ? __ffs(rej) - 1 : K;
        if (bad && tid <= acc && rank == 0) set_err(a.err, kErrToken);   // positions the walk reaches
        if (tid == 0) s_acc = acc;
    }
    __syncthreads();
    const int acc = s_acc;
    const float *pt = a.target + ((size_t)b * (K + 1) + acc) * V;
    const float u = uniform01(seed, 3, (uint32_t)b, (uint32_t)acc, 0);
    int extra = -1;
    if (acc < K) {
        const size_t row = (size_t)b * K + acc;
        const float *z = a.logits + row * V;
        const float lse = a.lse[row];
        extra = draw_cluster([&](int i) { return fmaxf(0.f, pt[i] - expf(z[i] * inv_t - lse)); }, V, u, sh);
    }
    if (extra < 0) extra = draw_cluster([&](int i) { return pt[i]; }, V, u, sh);
    if (rank == 0 && tid == 0) {
        a.accept_len[b] = acc;
        for (int j = 0; j <= K; ++j) {
            int v = -1;
            if (j < acc) v = a.draft[(size_t)b * K + j];
            else if (j == acc) v = extra;
            a.out_tokens[(size_t)b * (K + 1) + j] = v;
        }
        a.kv_len[b] += a.n_new[b];
    }
}

}  // namespace

int sample_blocks(int V, int *chunk) {
    int c = 2048;
    while ((V + c - 1) / c > kSampleMaxBlocks) c *= 2;
    if (chunk) *chunk = c;
    return (V + c - 1) / c;
}

cudaError_t launch_sample(const SampleArgs &args, int B, cudaStream_t s, bool pdl) {
    SampleArgs a = args;
    const int nblk = sample_blocks(a.V, &a.chunk);
    a.max_blocks = kSampleMaxBlocks;
    return launch_k(sample_kernel, dim3(nblk, B), dim3(kSampleThreads), 0, s, pdl, a);
}

cudaError_t launch_accept_sampled(const AcceptSampledArgs &a, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kAccCtas * a.B);
    cfg.blockDim = dim3(kAccThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kAccCtas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, accept_sampled_kernel, a);
}

}  // namespace prism
