// fp32 weight-streaming projections of the PRISM draft step (sm_103a).
//
// y[t] = W x[t] with W [rows, kin] in fp32 and a handful of activation rows:
// bound by reading W once from HBM, and at up to about 16 rows the CUDA cores
// keep up with that (fp32 has no tensor-core format that holds all its bits).
//   * An item is four rows of W (two gate/up pairs for SwiGLU).  A warp walks
//     the contraction of an item with its lanes side by side (16 bytes each)
//     and holds the item's 4 x TN sums in registers, so that one activation
//     vector read from shared memory serves four weight rows: reading it once
//     per weight row is what bounds a warp-per-row kernel (TN + 1 shared
//     reads per 4 TN multiply-adds, against TN + 4 per 16 TN here).
//   * Each lane copies its own weights into its warp's ring with cp.async and
//     reads back only what it copied: no barrier and no other thread between a
//     copy and its use, and the ring runs on across items.  The first copies
//     are issued before griddepcontrol.wait.
//   * The sums of an item are added over the lanes by a transposing butterfly
//     (31 shuffles for 32 sums instead of 160); each lane ends with one
//     output.
//   * With few items per SM, `seg` warps share an item's contraction and add
//     their sums in segment order; with more than 8 activation rows, `tg` warps
//     take 8 rows each of the same item.
//   * Small layers run as 8-warp CTAs of at most 110 KB, two to an SM, so that
//     the next projection's CTAs start and fill their rings while this one's
//     drain; layers with more bytes per SM as 16-warp CTAs with a larger ring
//     (small_layer has what either is worth).
//   * The LM head keeps the CTA's logits in shared memory, selects once per
//     chunk of units, publishes one list per row, and topk_merge_kernel joins
//     the CTAs' lists (the last CTA did that alone, with dependent loads).
// Gate/up + SwiGLU of one bf16 row takes the same kernel, on the row that the O
// projection's finish kernel wrote: the ring kernel spends 44 warp instructions on
// 512 bytes of weights, this one 16 (rounds of one sequence: 70B shape 3288 us
// there and 3099 here, 8B shape 1283 and 1279, 7B shape 987 and 982; on the tcgen05
// kernel the 8B shape took 1291 against 1281 on the ring kernel).
// A round of three sequences at hidden 1024, vocabulary 32000, K 4 (743 MB of
// weights): 741 us on the ring kernel that took fp32 before, 297 us here.
#include <algorithm>

#include "common.cuh"

namespace prism {

namespace {

constexpr int kMR = 4;                     // rows of W per item
constexpr int kF32MaxWarps = 16;
constexpr int kF32MaxRows = 32;            // activation rows of a pass (4 groups of 8)
constexpr int kNormVecs = 8;               // 16-byte vectors per lane of a row normalised in registers
constexpr int kStageBytes = kMR * 512;     // one k step of an item: 4 rows x 32 lanes x 16 bytes
constexpr size_t kF32Smem = 216 * 1024;    // dynamic shared memory of one CTA alone on an SM
constexpr size_t kF32SmemPair = 104 * 1024;  // of one of two
constexpr size_t kF32ZBytes = 32 * 1024;   // LM head: logits of one chunk

struct F32Plan {
    int warps;     // per CTA
    int tn, tg;    // activation rows per warp (1, 2, 4, 8), warps with different rows of one item
    int seg;       // warps that share an item's contraction
    int stages;    // ring stages per warp: 6, 4 or 2
    int chunk;     // LM head: items per selection chunk
    int prefetch;  // 1: request the next layer's first weights into L2
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint64_t pol) {
    if (pol)
        asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(pol) : "memory");
    else
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// All but the last S - 1 groups have landed.
__device__ __forceinline__ void cp_wait(int S) {
    if (S == 6) asm volatile("cp.async.wait_group 5;" ::: "memory");
    else if (S == 4) asm volatile("cp.async.wait_group 3;" ::: "memory");
    else asm volatile("cp.async.wait_group 1;" ::: "memory");
}
__device__ __forceinline__ void ffma2(unsigned long long &acc, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// A packed bf16 pair as two floats (exact).
__device__ __forceinline__ unsigned long long widen2(uint32_t w) {
    return ((unsigned long long)(w & 0xFFFF0000u) << 32) | (w << 16);
}

// The sums of N values over the 32 lanes: lane l ends with the sum of value
// l / (32 / N) (at each step a lane hands the half it does not keep to its
// partner; once one value is left, a plain butterfly).
template <int N>
__device__ __forceinline__ float reduce_transposed(float (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int n = N;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = lane & o;
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                if (i >= n) break;
                const float keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
                v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
            }
        } else {
            v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], o);
        }
    }
    return v[0];
}

__device__ __forceinline__ int clamp_new(const GemvArgs &a, int b) {
    const int n = a.n_new[b];
    if (n >= 1 && n <= a.max_new) return n;
    set_err(a.err, kErrNNew);
    return n < 1 ? 1 : a.max_new;
}
__device__ __forceinline__ int checked_token(const GemvArgs &a, int tok) {
    if (tok >= 0 && tok < a.vocab) return tok;
    set_err(a.err, kErrToken);
    return 0;
}

__device__ __forceinline__ void add_squares(float4 &q, const float4 &f) {
    q.x = fmaf(f.x, f.x, q.x);
    q.y = fmaf(f.y, f.y, q.y);
    q.z = fmaf(f.z, f.z, q.z);
    q.w = fmaf(f.w, f.w, q.w);
}
// 1 / RMS of a row from the lanes' sums of squares.
__device__ __forceinline__ float inv_rms(const float4 &q, const GemvArgs &a) {
    float ss = (q.x + q.y) + (q.z + q.w);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
    return 1.0f / sqrtf(ss / (float)a.d + a.eps);
}

// Activation rows t0 .. t0 + rows - 1 into X [rows][kin] (rows past a.T are
// zeros; bf16 rows are copied, and laid out as two planes).  The CTA's warps share the rows out; the warps of one row each sum
// its squares themselves, so that no barrier separates the norm's two halves.
template <typename WT>
__device__ __forceinline__ void stage_rows(const GemvArgs &a, int t0, int rows, float *X) {
    if constexpr (sizeof(WT) == 2) {
        const int nv = a.kin / 8;
        for (int e = threadIdx.x; e < rows * nv; e += blockDim.x) {
            const int r = e / nv, v = e % nv;
            const uint4 q = t0 + r < a.T ? __ldcg((const uint4 *)((const uint16_t *)a.act + (size_t)(t0 + r) * a.kin) + v)
                                         : make_uint4(0u, 0u, 0u, 0u);
            float4 *x = (float4 *)(X + (size_t)r * a.kin);
            x[v] = make_float4(bf16lo(q.x), bf16hi(q.x), bf16lo(q.y), bf16hi(q.y));
            x[nv + v] = make_float4(bf16lo(q.z), bf16hi(q.z), bf16lo(q.w), bf16hi(q.w));
        }
        return;
    }
    const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpr = rows < warps ? warps / rows : 1, share = warp % wpr;
    const int nvec = a.kin / 4, dv = a.d / 4;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int r = warp / wpr; r < rows; r += warps / wpr) {
        const int t = t0 + r;
        float4 *x = (float4 *)(X + (size_t)r * a.kin);
        const float4 *s0 = nullptr, *s1 = nullptr;       // elements below d, and from d on
        const float4 *g = nullptr;
        float inv = 1.f;
        if (t >= a.T) {
        } else if (a.pro == kProFusePrefill) {
            const int b = t / a.max_new, i = t % a.max_new;
            if (i < clamp_new(a, b)) {
                s0 = (const float4 *)((const float *)a.embed +
                                      (size_t)checked_token(a, a.tokens[b * a.max_new + i]) * a.d);
                s1 = (const float4 *)((const float *)a.hidden_in + ((size_t)b * a.max_new + i) * a.d);
            }
        } else if (a.pro == kProFuseDecode) {
            s0 = (const float4 *)((const float *)a.embed +
                                  (size_t)checked_token(a, a.draft[t * a.K + a.step - 2]) * a.d);
            s1 = (const float4 *)(a.src + (size_t)t * a.d);
        } else if (a.pro == kProNorm) {
            const int sr = a.src_prefill_rows ? t * a.max_new + clamp_new(a, t) - 1 : t;
            s0 = (const float4 *)(a.src + (size_t)sr * a.d);
            g = (const float4 *)a.gain;
            if (g && nvec <= kNormVecs * 32) {
                // the row in registers: one round trip for the sum and the values
                float4 f[kNormVecs];
#pragma unroll
                for (int i = 0; i < kNormVecs; ++i) f[i] = lane + 32 * i < nvec ? __ldcg(s0 + lane + 32 * i) : zero;
                float4 q = zero;
#pragma unroll
                for (int i = 0; i < kNormVecs; ++i) add_squares(q, f[i]);
                inv = inv_rms(q, a);
#pragma unroll
                for (int i = 0; i < kNormVecs; ++i) {
                    const int v = lane + 32 * i;
                    if (v >= nvec || i % wpr != share) continue;
                    const float4 w = __ldg(g + v);
                    x[v] = make_float4(f[i].x * inv * w.x, f[i].y * inv * w.y, f[i].z * inv * w.z, f[i].w * inv * w.w);
                }
                continue;
            }
            if (g) {
                float4 q = zero;
#pragma unroll 4
                for (int v = lane; v < nvec; v += 32) add_squares(q, __ldcg(s0 + v));
                inv = inv_rms(q, a);
            }
        } else {
            s0 = (const float4 *)((const float *)a.act + (size_t)t * a.kin);
        }
        const bool pair = s1 != nullptr;
#pragma unroll 8
        for (int v = share * 32 + lane; v < nvec; v += wpr * 32) {
            float4 f = !s0 ? zero : pair && v >= dv ? __ldcg(s1 + (v - dv)) : __ldcg(s0 + v);
            if (g) {
                const float4 w = __ldg(g + v);
                f = make_float4(f.x * inv * w.x, f.y * inv * w.y, f.z * inv * w.z, f.w * inv * w.w);
            }
            x[v] = f;
        }
    }
}

// TN: activation rows per warp.  RPW: rows of W per unit (2: gate and up).
template <typename WT, int TN, int RPW, bool TOPK>
__global__ void __launch_bounds__(kF32MaxWarps * 32, 1) gemv_rows4_kernel(const GemvArgs a, const F32Plan p) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    __shared__ float s_part[2][kF32MaxWarps][32];                  // segments' sums, double-buffered by item
    __shared__ Key s_list[TOPK ? kF32MaxRows : 1][kTopK];          // selections of the chunks so far
    constexpr int N = kMR * TN, UI = kMR / RPW, LPV = 32 / N;      // sums, units per item, lanes per sum
    constexpr int VEC = Elem<WT>::kPerVec;
    const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = p.stages, seg = p.seg, rows = p.tg * TN, nvec = a.kin / VEC;
    const int sg = warp % seg, tgi = warp / seg % p.tg, groups = warps / (seg * p.tg), grp = warp / (seg * p.tg);
    const int v_lo = (int)((long)sg * nvec / seg), v_hi = (int)((long)(sg + 1) * nvec / seg);
    const int nks = (v_hi - v_lo + 31) / 32;
    const int n_items = (a.n_units + UI - 1) / UI;
    const int i0 = (int)((long)blockIdx.x * n_items / gridDim.x), i1 = (int)((long)(blockIdx.x + 1) * n_items / gridDim.x);
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem_raw) + (uint32_t)(warp * S) * kStageBytes + lane * 16u;
    float *X = (float *)(smem_raw + (size_t)warps * S * kStageBytes);
    float *Z = X + (size_t)rows * a.kin;
    const int zs = p.chunk * UI;                                   // logits per row of a chunk
    const int n_pass = (a.T + rows - 1) / rows;
    // W is read once per pass: with several, the later ones should find it in L2
    const uint64_t pol = a.w_evict_first && n_pass == 1 ? l2_evict_first_policy() : 0ull;
    pdl_trigger();

    // the copies of this warp, stepped: item, k step, ring slot
    int ci = 0, cks = 0, cslot = 0, cend = 0;
    auto copy_next = [&]() {
        if (ci < cend) {
            const int v = v_lo + cks * 32 + lane;
            if (v < v_hi) {
                const WT *w = (const WT *)a.W + (size_t)v * VEC;
#pragma unroll
                for (int r = 0; r < kMR; ++r) {
                    const int u = min(ci * UI + r % UI, a.n_units - 1) + (r / UI) * a.pair_offset;
                    cp_async16(ring + (uint32_t)cslot * kStageBytes + r * 512u, w + (size_t)u * a.kin, pol);
                }
            }
            if (++cks == nks) { cks = 0; ci += groups; }
        }
        cp_commit();
        if (++cslot == S) cslot = 0;
    };
    auto start_copies = [&](int c0, int c1) {
        ci = c0 + grp;
        cks = cslot = 0;
        cend = c1;
        for (int s = 0; s < S; ++s) copy_next();
    };

    const int per_chunk = TOPK ? p.chunk : max(i1 - i0, 1);
    start_copies(i0, min(i0 + per_chunk, i1));
    // the gain is a weight: requested early, it is in L2 when the rows are normalised
    if (a.pro == kProNorm && a.gain && threadIdx.x * 32 < a.d)
        asm volatile("prefetch.global.L2 [%0];" ::"l"((const float *)a.gain + threadIdx.x * 32) : "memory");
    pdl_wait();

    for (int pass = 0; pass < n_pass; ++pass) {
        const int t0 = pass * rows, tc = min(rows, a.T - t0);
        if (pass) __syncthreads();
        stage_rows<WT>(a, t0, rows, X);
        __syncthreads();
        int c0 = i0;
        do {
            const int c1 = min(c0 + per_chunk, i1);
            if (pass || c0 != i0) start_copies(c0, c1);
            int slot = 0, buf = 0;
            for (int it = c0 + grp; it < c1; it += groups) {
                unsigned long long acc[kMR][TN];
#pragma unroll
                for (int r = 0; r < kMR; ++r)
#pragma unroll
                    for (int t = 0; t < TN; ++t) acc[r][t] = 0ull;
                for (int ks = 0; ks < nks; ++ks) {
                    cp_wait(S);
                    const int v = v_lo + ks * 32 + lane;
                    if (v < v_hi) {
                        ulonglong2 w[kMR];
#pragma unroll
                        for (int r = 0; r < kMR; ++r)
                            asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(w[r].x), "=l"(w[r].y)
                                         : "r"(ring + (uint32_t)slot * kStageBytes + r * 512u) : "memory");
                        const ulonglong2 *x = (const ulonglong2 *)(X + (size_t)(tgi * TN) * a.kin) + v;
#pragma unroll
                        for (int t = 0; t < TN; ++t) {
                            if constexpr (VEC == 4) {
                                const ulonglong2 xv = x[(size_t)t * nvec];
#pragma unroll
                                for (int r = 0; r < kMR; ++r) {
                                    ffma2(acc[r][t], w[r].x, xv.x);
                                    ffma2(acc[r][t], w[r].y, xv.y);
                                }
                            } else {
                                // eight weights, widened exactly; X holds the first and the last
                                // four of every eight activations as two planes (no bank conflicts)
                                const ulonglong2 xa = x[(size_t)t * 2 * nvec], xb = x[(size_t)t * 2 * nvec + nvec];
#pragma unroll
                                for (int r = 0; r < kMR; ++r) {
                                    ffma2(acc[r][t], widen2((uint32_t)w[r].x), xa.x);
                                    ffma2(acc[r][t], widen2((uint32_t)(w[r].x >> 32)), xa.y);
                                    ffma2(acc[r][t], widen2((uint32_t)w[r].y), xb.x);
                                    ffma2(acc[r][t], widen2((uint32_t)(w[r].y >> 32)), xb.y);
                                }
                            }
                        }
                    }
                    if (++slot == S) slot = 0;
                    copy_next();
                }
                float sums[N];                                     // sum t * 4 + r
#pragma unroll
                for (int t = 0; t < TN; ++t)
#pragma unroll
                    for (int r = 0; r < kMR; ++r)
                        sums[t * kMR + r] = __uint_as_float((uint32_t)acc[r][t]) + __uint_as_float((uint32_t)(acc[r][t] >> 32));
                float z = reduce_transposed<N>(sums);
                const int idx = lane / LPV;
                if (seg > 1) {
                    if (lane % LPV == 0) s_part[buf][warp][idx] = z;
                    asm volatile("bar.sync %0, %1;" ::"r"(1 + warp / seg), "r"(seg * 32) : "memory");
                    const int b = buf;
                    buf ^= 1;
                    if (sg != 0) continue;
                    z = s_part[b][warp][idx];
                    for (int q = 1; q < seg; ++q) z += s_part[b][warp + q][idx];
                }
                const float up = RPW == 2 ? __shfl_down_sync(0xFFFFFFFFu, z, UI * LPV) : 0.f;
                const int r = idx % kMR, tl = tgi * TN + idx / kMR, t = t0 + tl, u = it * UI + r;
                if (lane % LPV != 0 || r >= UI || tl >= tc || u >= a.n_units) continue;
                if constexpr (TOPK) {
                    if (a.logits) a.logits[((size_t)t * a.K + a.step - 1) * a.vocab + u] = z;
                    Z[(size_t)tl * zs + (u - c0 * UI)] = z;
                } else if constexpr (RPW == 2) {
                    Elem<WT>::store((WT *)a.out_act, (size_t)t * a.out_ld + u, z / (1.0f + expf(-z)) * up);
                } else {
                    if (a.epi == kEpiResid) {
                        z += a.resid[(size_t)(a.resid_prefill_rows ? t * a.max_new + clamp_new(a, t) - 1 : t) * a.out_ld + u];
                        if (a.hidden_out) a.hidden_out[((size_t)t * a.K + a.step - 1) * a.d + u] = z;
                    }
                    a.out[(size_t)t * a.out_ld + u] = z;
                }
            }
            if constexpr (TOPK) {
                __syncthreads();
                const int n = min(c1 * UI, a.n_units) - c0 * UI;
                for (int tl = warp; tl < tc; tl += warps) {
                    // below every candidate, and what an empty place of a list reads as
                    const Key none = pack_best(-INFINITY, 0x7FFFFFFF);
                    Key l[kTopK];
#pragma unroll
                    for (int i = 0; i < kTopK; ++i) l[i] = c0 != i0 && lane == 0 ? s_list[tl][i] : none;
                    for (int j = lane; j < n; j += 32) {
                        const float z = Z[(size_t)tl * zs + j];
                        if (z == z) key_insert(l, pack_best(z + 0.f, c0 * UI + j));   // NaN is no candidate, -0 equals 0
                    }
#pragma unroll 1
                    for (int m = 1; m < 32; m <<= 1) key_merge_xor(l, m);
                    if (lane < kTopK) {
                        const Key k = key_at(l, lane);
                        if (c1 < i1) {
                            s_list[tl][lane] = k;
                        } else {
                            float v;
                            int id;
                            unpack_best(k, v, id);
                            const size_t o = ((size_t)(t0 + tl) * gridDim.x + blockIdx.x) * kTopK + lane;
                            a.lm_part[o] = v;
                            a.lm_part_id[o] = id;
                        }
                    }
                }
                if (c1 < i1) __syncthreads();
            }
            c0 = c1;
        } while (c0 < i1);
    }
    if (p.prefetch && threadIdx.x == 0) prefetch_l2_share(a.pf_next, a.pf_next_bytes, blockIdx.x, gridDim.x);
}

template <int TN>
cudaError_t dispatch_f32(const GemvArgs &a, const F32Plan &p, int grid, size_t smem, cudaStream_t s, bool pdl) {
    const dim3 g(grid), b(p.warps * 32);
    if (a.epi == kEpiTopK) return launch_k(gemv_rows4_kernel<float, TN, 1, true>, g, b, smem, s, pdl, a, p);
    if (a.epi == kEpiSwiGLU) return launch_k(gemv_rows4_kernel<float, TN, 2, false>, g, b, smem, s, pdl, a, p);
    return launch_k(gemv_rows4_kernel<float, TN, 1, false>, g, b, smem, s, pdl, a, p);
}

template <int TN>
cudaError_t f32_attrs() {
    cudaError_t e = cudaFuncSetAttribute(gemv_rows4_kernel<float, TN, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kF32Smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gemv_rows4_kernel<float, TN, 2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kF32Smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gemv_rows4_kernel<float, TN, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kF32Smem);
    return e;
}

// A layer with fewer bytes per CTA than this runs as 8-warp CTAs, two to an SM, and
// makes no L2 requests for the next; a bf16 gate/up row of such a layer stays on the
// ring kernel.  The line was drawn between hidden 1024 (up to 160 KB per CTA outside the
// LM head) and 4096 (450 KB and more).  Both sides of it since (K 4, vocabulary
// 32000, contexts of 200, us a round; every layer as 16-warp CTAs in brackets), fp32 rounds of
// 1 / 3 / 12 sequences: hidden 256 161 / 184 / 377 (170 / 172 / 284), 1024 256 / 320 / 620
// (252 / 296 / 539), 2048 443 / 540 / 1141 (421 / 494 / 1048), 3072 685 / 842 / 2046 (675 /
// 822 / 2022), 4096 the same: the 8-warp CTAs pay for one sequence at hidden 256 alone.
// One bf16 sequence on the ring kernel and on this one: hidden 1024 201 and 195 us, 1536 233
// and 232, 2048 with 304 KB per CTA 287 and 283, with 432 KB 307 and 299, 3072 397 and 390,
// 4096 562 and 560: nowhere a loss since small layers' L2 requests went (198 and 207 before).
bool small_layer(const GemvArgs &a, int es, int grid) {
    const int UI = a.epi == kEpiSwiGLU ? kMR / 2 : kMR;
    const int n_items = (a.n_units + UI - 1) / UI, per_cta = (n_items + grid - 1) / grid;
    return (size_t)per_cta * kMR * a.kin * es < 384 * 1024;
}

// The most activation rows per pass that fit beside the smallest ring, then
// the largest ring; then the segment count with the shortest run of k steps.
bool f32_plan(const GemvArgs &a, int es, int grid, F32Plan &p, size_t &smem) {
    const int UI = a.epi == kEpiSwiGLU ? kMR / 2 : kMR;
    const int n_items = (a.n_units + UI - 1) / UI, per_cta = (n_items + grid - 1) / grid;
    const bool small = small_layer(a, es, grid);
    // beside such CTAs the next layer's own rings are already filling: requests
    // for its first bytes only delay them (three sequences at hidden 1024, on the build
    // of that step: 339 us a round with, 327 without)
    p.prefetch = !small;
    p.tn = a.T <= 1 ? 1 : a.T <= 2 ? 2 : a.T <= 4 ? 4 : 8;
    p.tg = a.T <= 8 ? 1 : a.T <= 16 ? 2 : 4;
    for (;;) {
        const int rows = p.tn * p.tg;
        p.chunk = a.epi == kEpiTopK ? std::min(per_cta, (int)(kF32ZBytes / 4 / rows / UI)) : 0;
        const size_t x = (size_t)rows * a.kin * 4 + (size_t)p.chunk * UI * rows * 4;
        for (size_t room : {kF32SmemPair, kF32Smem}) {
            if (room == kF32SmemPair && !small) continue;
            p.warps = room == kF32SmemPair || (small && p.tg == 1) ? 8 : 16;
            for (int S : {6, 4, 2})
                if ((smem = (size_t)p.warps * S * kStageBytes + x) <= room) {
                    p.stages = S;
                    const int nk = (a.kin * es / 16 + 31) / 32;
                    long best = -1;
                    for (int seg = 1; seg * p.tg <= p.warps && seg <= nk; seg *= 2) {
                        const int groups = p.warps / (seg * p.tg);
                        const long cost = (long)((per_cta + groups - 1) / groups) * ((nk + seg - 1) / seg + 1);
                        if (best < 0 || cost < best) { best = cost; p.seg = seg; }
                    }
                    return true;
                }
        }
        if (p.tg > 1) p.tg /= 2;
        else if (p.tn > 1) p.tn /= 2;
        else return false;
    }
}

}  // namespace

cudaError_t prepare_gemv_f32_kernels() {
    cudaError_t e = f32_attrs<1>();
    if (e == cudaSuccess) e = f32_attrs<2>();
    if (e == cudaSuccess) e = f32_attrs<4>();
    if (e == cudaSuccess) e = f32_attrs<8>();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gemv_rows4_kernel<uint16_t, 1, 2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kF32Smem);
    return e;
}

bool gemv_pair_supported(const GemvArgs &a, int grid) {
    F32Plan p{};
    size_t smem;
    // (a small layer stays on the ring kernel, which norms its row itself; see small_layer)
    return a.epi == kEpiSwiGLU && a.T == 1 && !small_layer(a, 2, grid) && f32_plan(a, 2, grid, p, smem);
}

cudaError_t launch_gemv_pair(const GemvArgs &a, int grid, cudaStream_t s, bool pdl) {
    F32Plan p{};
    size_t smem;
    if (a.pro != kProCopy || !gemv_pair_supported(a, grid) || !f32_plan(a, 2, grid, p, smem)) return cudaErrorInvalidValue;
    p.prefetch = 1;
    return launch_k(gemv_rows4_kernel<uint16_t, 1, 2, false>, dim3(grid), dim3(p.warps * 32), smem, s, pdl, a, p);
}

cudaError_t launch_gemv_f32(const GemvArgs &a, int grid, cudaStream_t s, bool pdl) {
    F32Plan p{};
    size_t smem;
    if (!f32_plan(a, 4, grid, p, smem)) return cudaErrorInvalidValue;
    cudaError_t e = p.tn == 1   ? dispatch_f32<1>(a, p, grid, smem, s, pdl)
                    : p.tn == 2 ? dispatch_f32<2>(a, p, grid, smem, s, pdl)
                    : p.tn == 4 ? dispatch_f32<4>(a, p, grid, smem, s, pdl)
                                : dispatch_f32<8>(a, p, grid, smem, s, pdl);
    if (e == cudaSuccess && a.epi == kEpiTopK && !a.defer_merge) e = launch_topk_merge(a, grid, s);
    return e;
}

}  // namespace prism
