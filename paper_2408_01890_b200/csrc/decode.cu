// Decode step of a shared layer (Sec. 5.2, decoding stage) and of a standard layer (Eq. 1-2, last row).
//
// Both are streaming scans over a cache, bound by HBM bandwidth.  Work is split over (sequence b, chunk of cached positions, and
// for small batches groups of heads); the scores of a shared layer's chunk need the previous layer's scores of ALL heads
// because the aligner mixes them:
//   phase A  scores of the chunk for every head
//            shared:   A[:,j] = W2^T act(W1^T prev[:,j] + b1) + b2 + q'.K'_j/sqrt(r)     (Eq. 3-4)
//            standard: A[h,j] = q_h.K_j/sqrt(d)                                           (Eq. 2)
//            and, if asked, the row handed to the next shared layer
//   phase B  chunk-local softmax statistics (max, sum) per head and the partial product with V
// A second kernel merges the per-chunk partials (m, l, o) into the output (split-K softmax).
// K' is cached transposed ([r][L_cap], position contiguous) so that r = 21 needs no padding and every
// load is a full 16-byte vector along the position axis; V rows are 256 contiguous bytes.
// bf16 caches of head width 128 (32 or 40 heads for a shared layer) run on the kernels of decode_fast.cuh; the kernels here
// take every other head count, width, type and Integrate mode.
#include <algorithm>
#include <climits>

#include "decode_fast.cuh"

namespace lisa {
namespace {

constexpr int kChunk = 128;
constexpr int kThreads = kDecodeThreads;
constexpr int kWarps = kDecodeWarps;

// Partial P.V of a FULL chunk (all kChunk rows valid), bf16 cache, LPR = d/8 lanes per V row (general kernels, d < 128).  A warp streams the
// V rows of its heads as one software-pipelined sequence: two register sets of eight 16-byte loads per lane
// alternate, and the last batch of a head already prefetches the first batch of the warp's next head, so loads
// stay in flight across batches and across heads.  All offsets are compile-time constants off one pointer.
template <int LPR>
__device__ __forceinline__ void pv_full_chunk(const DecodeParams& p, const float* s_s, int b, size_t part, int j0) {
    constexpr int RSTEP = 32 / LPR;            // rows fetched by one warp-wide load
    constexpr int NB = kChunk / RSTEP / 8;     // batches of 8 loads per head (even)
    constexpr int D = LPR * 8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane % LPR, rsel = lane / LPR;
    const int Hq = p.Hq, G = p.Hq / p.Hkv;
    auto head_ptr = [&](int h) {
        return reinterpret_cast<const uint4*>(p.vcache) + (((size_t)b * p.Hkv + h / G) * p.L_cap + j0 + rsel) * LPR + sub;
    };
    if (warp >= Hq) return;
    const uint4* hp = head_ptr(warp);
    uint4 ra[8], rb[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) ra[u] = ld_stream16(hp + u * RSTEP * LPR);
    for (int h = warp; h < Hq; h += kWarps) {
        const bool has_next = h + kWarps < Hq;
        const uint4* np = has_next ? head_ptr(h + kWarps) : hp;
        const float* ps = s_s + h * kChunk + rsel;
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int bi = 0; bi < NB; bi += 2) {
#pragma unroll
            for (int u = 0; u < 8; ++u) rb[u] = ld_stream16(hp + ((bi + 1) * 8 + u) * RSTEP * LPR);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                float f[8];
                bf16x8_to_f32(ra[u], f);
                const float pj = ps[(bi * 8 + u) * RSTEP];
#pragma unroll
                for (int t = 0; t < 8; ++t) acc[t] = fmaf(pj, f[t], acc[t]);
            }
            if (bi + 2 < NB) {
#pragma unroll
                for (int u = 0; u < 8; ++u) ra[u] = ld_stream16(hp + ((bi + 2) * 8 + u) * RSTEP * LPR);
            } else if (has_next) {
#pragma unroll
                for (int u = 0; u < 8; ++u) ra[u] = ld_stream16(np + u * RSTEP * LPR);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                float f[8];
                bf16x8_to_f32(rb[u], f);
                const float pj = ps[((bi + 1) * 8 + u) * RSTEP];
#pragma unroll
                for (int t = 0; t < 8; ++t) acc[t] = fmaf(pj, f[t], acc[t]);
            }
        }
#pragma unroll
        for (int off = LPR; off < 32; off <<= 1)
#pragma unroll
            for (int t = 0; t < 8; ++t) acc[t] += __shfl_xor_sync(0xffffffffu, acc[t], off);
        if (rsel == 0) {
            float4* dst = reinterpret_cast<float4*>(p.ws_o + (part + h) * D + sub * 8);
            dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
            dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
        }
        hp = np;
    }
}

// ---------------------------------------------------------------------------------------------
// Phase B: s_s[h][kChunk] holds the chunk's scores (-inf beyond the sequence end). Produces the
// chunk's (max, sum, unnormalised P.V) per head into the workspace.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void softmax_pv_chunk(const DecodeParams& p, float* s_s, int b, int chunk, int nrows) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Hq = p.Hq, d = p.d, G = p.Hq / p.Hkv;
    const size_t part = ((size_t)b * p.n_chunks + chunk) * Hq;
    for (int h = warp; h < Hq; h += kWarps) {
        float v[kChunk / 32];
        float cmax = -INFINITY;
#pragma unroll
        for (int t = 0; t < kChunk / 32; ++t) {
            v[t] = s_s[h * kChunk + lane + 32 * t];
            cmax = fmaxf(cmax, v[t]);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, off));
        float sum = 0.f;
#pragma unroll
        for (int t = 0; t < kChunk / 32; ++t) {
            const float e = __expf(v[t] - cmax);
            s_s[h * kChunk + lane + 32 * t] = e;
            sum += e;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
        if (lane == 0) {
            p.ws_m[part + h] = cmax;
            p.ws_l[part + h] = sum;
        }
    }
    __syncthreads();
    const int j0 = chunk * kChunk;
    if (p.cache_dtype == LISA_BF16) {
        if (nrows == kChunk) {
            if (d == 128) pv_full_chunk<16>(p, s_s, b, part, j0);
            else if (d == 64) pv_full_chunk<8>(p, s_s, b, part, j0);
            else pv_full_chunk<4>(p, s_s, b, part, j0);
        } else {
            // ragged last chunk of a sequence: plain loop
            const int lpr = d / 8, rstep = 32 / lpr, sub = lane % lpr, rsel = lane / lpr;
            for (int h = warp; h < Hq; h += kWarps) {
                const uint4* vbase = reinterpret_cast<const uint4*>(p.vcache) +
                                     (((size_t)b * p.Hkv + h / G) * p.L_cap + j0) * lpr + sub;
                const float* ps = s_s + h * kChunk;
                float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                for (int jj = rsel; jj < nrows; jj += rstep) {
                    float f[8];
                    bf16x8_to_f32(ld_stream16(vbase + (size_t)jj * lpr), f);
                    const float pj = ps[jj];
#pragma unroll
                    for (int t = 0; t < 8; ++t) acc[t] = fmaf(pj, f[t], acc[t]);
                }
                for (int off = lpr; off < 32; off <<= 1)
#pragma unroll
                    for (int t = 0; t < 8; ++t) acc[t] += __shfl_xor_sync(0xffffffffu, acc[t], off);
                if (rsel == 0) {
                    float4* dst = reinterpret_cast<float4*>(p.ws_o + (part + h) * d + sub * 8);
                    dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
                    dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
                }
            }
        }
    } else {
        // fp32 cache: thread per output column
        for (int e = tid; e < Hq * d; e += kThreads) {
            const int h = e / d, x = e % d;
            const float* vb = reinterpret_cast<const float*>(p.vcache) + (((size_t)b * p.Hkv + h / G) * p.L_cap + j0) * d + x;
            float acc = 0.f;
            for (int jj = 0; jj < nrows; ++jj) acc = fmaf(s_s[h * kChunk + jj], vb[(size_t)jj * d], acc);
            p.ws_o[(part + h) * d + x] = acc;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Shared layer: any supported mode and size, thread per position with per-thread scratch arrays.
// ---------------------------------------------------------------------------------------------
template <bool RB>
__global__ void __launch_bounds__(kThreads, 1) shared_decode_chunk_kernel(const __grid_constant__ DecodeParams p) {
    extern __shared__ __align__(16) float smem[];
    const int b = blockIdx.y, chunk = blockIdx.x, tid = threadIdx.x;
    chain_release();
    const int j0 = chunk * kChunk;
    const int Hq = p.Hq;
    const int m = p.integrate == LISA_INTEGRATE_PLUS ? 0 : p.m;
    const int r = p.r, G = Hq / p.Hkv;
    const int h_in = p.integrate == LISA_INTEGRATE_CONCAT ? 2 * Hq : Hq;

    float* s_s = smem;                      // [Hq][kChunk]  delta, then scores, then exp
    float* qp_s = s_s + Hq * kChunk;        // [Hq][kMaxRank]
    float* w1_s = qp_s + Hq * kMaxRank;     // [h_in][m]
    float* w2_s = w1_s + h_in * m;          // [m][Hq]
    float* b1_s = w2_s + m * Hq;            // [m]
    float* b2_s = b1_s + m;                 // [Hq]

    // the aligner's weights are constants of the model: staged while the kernel before this one may still be running
    if (p.integrate != LISA_INTEGRATE_PLUS) {
        for (int e = tid; e < h_in * m; e += kThreads) w1_s[e] = ld_elem(p.w1, e, p.w_dtype);
        for (int e = tid; e < m; e += kThreads) b1_s[e] = ldw(p.b1, e, p.w_dtype);
        if (p.ffn_layers == 2) {
            for (int e = tid; e < m * Hq; e += kThreads) w2_s[e] = ld_elem(p.w2, e, p.w_dtype);
            for (int e = tid; e < Hq; e += kThreads) b2_s[e] = ldw(p.b2, e, p.w_dtype);
        }
    }
    chain_wait();   // from here on: lengths, Q', the caches and the score row, which earlier kernels of the stream produce
    const int L = decode_length(p, b);
    if (j0 >= L) return;
    const int nrows = min(kChunk, L - j0);
    for (int e = tid; e < Hq * r; e += kThreads) {
        const int h = e / r, x = e % r;
        qp_s[h * kMaxRank + x] = ld_elem(p.qp.ptr, b * p.qp.sb + h * p.qp.sh + x, p.qp.dtype);
    }
    __syncthreads();

    // A_Delta for the chunk (Eq. 3): unit = (head, 8 consecutive positions)
    const float inv_sqrt_r = rsqrtf((float)r);
    if (p.cache_dtype == LISA_BF16) {
        for (int u = tid; u < Hq * (kChunk / 8); u += kThreads) {
            const int h = u / (kChunk / 8), j8 = u % (kChunk / 8);
            float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (j0 + j8 * 8 < p.L_cap) {
                const __nv_bfloat16* base = reinterpret_cast<const __nv_bfloat16*>(p.kpT) +
                                            ((size_t)b * p.Hkv + h / G) * r * p.L_cap + j0 + j8 * 8;
                for (int x0 = 0; x0 < r; x0 += 8) {   // eight independent 16-byte loads in flight per lane
                    uint4 raw[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        raw[e] = x0 + e < r ? ld_stream16(base + (size_t)(x0 + e) * p.L_cap) : make_uint4(0, 0, 0, 0);
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        float f[8];
                        bf16x8_to_f32(raw[e], f);
                        const float qx = x0 + e < r ? qp_s[h * kMaxRank + x0 + e] : 0.f;
#pragma unroll
                        for (int t = 0; t < 8; ++t) acc[t] = fmaf(qx, f[t], acc[t]);
                    }
                }
            }
            float4* dst = reinterpret_cast<float4*>(s_s + h * kChunk + j8 * 8);
            dst[0] = make_float4(acc[0] * inv_sqrt_r, acc[1] * inv_sqrt_r, acc[2] * inv_sqrt_r, acc[3] * inv_sqrt_r);
            dst[1] = make_float4(acc[4] * inv_sqrt_r, acc[5] * inv_sqrt_r, acc[6] * inv_sqrt_r, acc[7] * inv_sqrt_r);
        }
    } else {
        for (int u = tid; u < Hq * kChunk; u += kThreads) {
            const int h = u / kChunk, jj = u % kChunk;
            float acc = 0.f;
            if (jj < nrows) {
                const float* base = reinterpret_cast<const float*>(p.kpT) + ((size_t)b * p.Hkv + h / G) * r * p.L_cap + j0 + jj;
                for (int x = 0; x < r; ++x) acc = fmaf(qp_s[h * kMaxRank + x], base[(size_t)x * p.L_cap], acc);
            }
            s_s[u] = acc * inv_sqrt_r;
        }
    }
    __syncthreads();

    const int pos = tid & (kChunk - 1), half = tid / kChunk;
    const bool valid = pos < nrows;
    const int64_t prev_i = b * p.prev_sb + j0 + pos;     // this thread's position in the previous layer's row of head 0
    const int64_t out_i = b * p.sc_sb + j0 + pos;

    {
        if (half == 0) {
            float a[kMaxHeads], dl[kMaxHeads], hid[kMaxHidden];
            for (int h = 0; h < Hq; ++h) {
                a[h] = valid ? ld_row<RB>(p.prev, prev_i + h * p.prev_sh) : 0.f;
                dl[h] = s_s[h * kChunk + pos];
            }
            if (p.integrate == LISA_INTEGRATE_PLUS) {
                for (int g = 0; g < Hq; ++g) a[g] += dl[g];
            } else {
                for (int u = 0; u < m; ++u) {
                    float s = b1_s[u];
                    for (int x = 0; x < Hq; ++x) s = fmaf(a[x], w1_s[x * m + u], s);
                    if (p.integrate == LISA_INTEGRATE_CONCAT)
                        for (int x = 0; x < Hq; ++x) s = fmaf(dl[x], w1_s[(Hq + x) * m + u], s);
                    hid[u] = s;
                }
                if (p.ffn_layers == 1) {
                    for (int g = 0; g < Hq; ++g) a[g] = hid[g];
                } else {
                    for (int u = 0; u < m; ++u) hid[u] = act_apply(hid[u], p.act);
                    for (int g = 0; g < Hq; ++g) {
                        float s = b2_s[g];
                        for (int u = 0; u < m; ++u) s = fmaf(hid[u], w2_s[u * Hq + g], s);
                        a[g] = s;
                    }
                }
                if (p.integrate == LISA_INTEGRATE_ADD)
                    for (int g = 0; g < Hq; ++g) a[g] += dl[g];
            }
            for (int g = 0; g < Hq; ++g) {
                s_s[g * kChunk + pos] = valid ? a[g] : -INFINITY;
                if (valid && p.out_scores) st_row<RB>(p.out_scores, out_i + g * p.sc_sh, a[g]);
            }
        }
    }
    __syncthreads();
    softmax_pv_chunk(p, s_s, b, chunk, nrows);
}

// ---------------------------------------------------------------------------------------------
// Standard layer: scores from the K cache.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads, 2) anchor_decode_chunk_kernel(const __grid_constant__ DecodeParams p) {
    extern __shared__ __align__(16) float smem[];
    const int b = blockIdx.y, chunk = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    chain_release();
    chain_wait();
    const int L = decode_length(p, b);
    const int j0 = chunk * kChunk;
    if (j0 >= L) return;
    const int nrows = min(kChunk, L - j0);
    const int Hq = p.Hq, d = p.d, G = Hq / p.Hkv;
    float* s_s = smem;               // [Hq][kChunk]
    float* q_s = s_s + Hq * kChunk;  // [Hq][d]
    for (int e = tid; e < Hq * d; e += kThreads) {
        const int h = e / d, x = e % d;
        q_s[e] = ld_elem(p.q.ptr, b * p.q.sb + h * p.q.sh + x, p.q.dtype);
    }
    __syncthreads();
    const float inv_sqrt_d = rsqrtf((float)d);
    if (p.cache_dtype == LISA_BF16) {
        const int lpr = d / 8, rstep = 32 / lpr, sub = lane % lpr, rsel = lane / lpr;
        for (int h = warp; h < Hq; h += kWarps) {
            float qv[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) qv[t] = q_s[h * d + sub * 8 + t];
            const uint4* kbase = reinterpret_cast<const uint4*>(p.kcache) +
                                 (((size_t)b * p.Hkv + h / G) * p.L_cap + j0) * lpr + sub;
            for (int jb = 0; jb < kChunk; jb += 4 * rstep) {
                float dot[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int jj = jb + u * rstep + rsel;
                    dot[u] = 0.f;
                    if (jj < nrows) {
                        float f[8];
                        bf16x8_to_f32(ld_stream16(kbase + (size_t)jj * lpr), f);
#pragma unroll
                        for (int t = 0; t < 8; ++t) dot[u] = fmaf(qv[t], f[t], dot[u]);
                    }
                }
                for (int off = lpr >> 1; off > 0; off >>= 1)
#pragma unroll
                    for (int u = 0; u < 4; ++u) dot[u] += __shfl_xor_sync(0xffffffffu, dot[u], off);
                if (sub == 0) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int jj = jb + u * rstep + rsel;
                        if (jj < kChunk) s_s[h * kChunk + jj] = jj < nrows ? dot[u] * inv_sqrt_d : -INFINITY;
                    }
                }
            }
        }
    } else {
        for (int u = tid; u < Hq * kChunk; u += kThreads) {
            const int h = u / kChunk, jj = u % kChunk;
            float acc = -INFINITY;
            if (jj < nrows) {
                const float* kr = reinterpret_cast<const float*>(p.kcache) + (((size_t)b * p.Hkv + h / G) * p.L_cap + j0 + jj) * d;
                acc = 0.f;
                for (int x = 0; x < d; ++x) acc = fmaf(q_s[h * d + x], kr[x], acc);
                acc *= inv_sqrt_d;
            }
            s_s[u] = acc;
        }
    }
    __syncthreads();
    if (p.out_scores) {
        for (int u = tid; u < Hq * kChunk; u += kThreads) {
            const int h = u / kChunk, jj = u % kChunk;
            if (jj < nrows) {
                if (p.row_bf16) st_row<true>(p.out_scores, b * p.sc_sb + h * p.sc_sh + j0 + jj, s_s[u]);
                else st_row<false>(p.out_scores, b * p.sc_sb + h * p.sc_sh + j0 + jj, s_s[u]);
            }
        }
    }
    softmax_pv_chunk(p, s_s, b, chunk, nrows);
}

// Merge the per-chunk (m, l, o) partials of one (b, h): o = sum_c e^{m_c - M} o_c / sum_c e^{m_c - M} l_c.  Bound by latency: every
// warp forms M and the denominator by itself (the chunks' m and l come from L2), its lanes take four columns each, the warps
// different chunks, and one exchange through shared memory adds their sums; a thread's first U partial outputs come with the maxima, not
// behind them (with the chunk kernels' q' loads in flight together: one layer of the paper's default model, 8 x 1111, 38.9 -> 35.2 us;
// 7B-shaped, 1 x 333, 12.0 -> 11.2; 13B-shaped, 64 x 4096, 518 -> 515).
// U outputs, as many as a thread has where the contexts are short (38 sequences of 180 positions, anchor and three layers: 101 us with one or two,
// 107 with eight), and no more than leave the grid resident at once: with eight an SM holds 8 CTAs of 64 registers a thread, with two 10, with
// one 12 (anchor and three layers of 8 KV heads, us, with eight | one: 100 sequences of up to 1150 positions, four fifths of them short, 182 | 172;
// all of 1150 422 | 416; 60 of 1250, 40 heads 841 | 838; 40 of 1000, where two are resident and one is not needed, with two | one 187 | 190).
constexpr int kMergeThreads = 128;
template <int U>
__global__ void __launch_bounds__(kMergeThreads) decode_merge_kernel(const __grid_constant__ DecodeParams p) {
    __shared__ float4 s_o[kMergeThreads];
    const int h = blockIdx.x, b = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
    if (!p.late_release) chain_release();
    chain_wait();
    if (p.late_release) chain_release();
    const int nc = (decode_length(p, b) + p.chunk - 1) / p.chunk;
    const size_t base = (size_t)b * p.n_chunks * p.Hq + h;
    const int lpr = p.d / 4, x = tid % lpr, c0 = tid / lpr, cstep = kMergeThreads / lpr;   // lanes per partial output, this thread's chunks
    const float4* po = reinterpret_cast<const float4*>(p.ws_o + base * p.d) + x;
    const size_t step = (size_t)p.Hq * lpr;
    float4 first[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (c0 + u * cstep < nc) first[u] = po[(size_t)(c0 + u * cstep) * step];
    float M = -INFINITY;
    for (int c = lane; c < nc; c += 32) M = fmaxf(M, p.ws_m[base + (size_t)c * p.Hq]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    float den = 0.f;
    for (int c = lane; c < nc; c += 32) den = fmaf(__expf(p.ws_m[base + (size_t)c * p.Hq] - M), p.ws_l[base + (size_t)c * p.Hq], den);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    auto add = [&](int c, const float4& o) {
        const float w = __expf(p.ws_m[base + (size_t)c * p.Hq] - M);
        acc.x = fmaf(w, o.x, acc.x); acc.y = fmaf(w, o.y, acc.y); acc.z = fmaf(w, o.z, acc.z); acc.w = fmaf(w, o.w, acc.w);
    };
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (c0 + u * cstep < nc) add(c0 + u * cstep, first[u]);
#pragma unroll 8
    for (int c = c0 + U * cstep; c < nc; c += cstep) add(c, po[(size_t)c * step]);
    s_o[tid] = acc;
    __syncthreads();
    if (tid >= lpr) return;
    for (int q = 1; q < cstep; ++q) {
        const float4 o = s_o[q * lpr + tid];
        acc.x += o.x; acc.y += o.y; acc.z += o.z; acc.w += o.w;
    }
    const float inv = 1.f / den;
    const int64_t at = b * p.o.sb + h * p.o.sh + 4 * tid;
    void* out = const_cast<void*>(p.o.ptr);
    st_elem(out, at, p.o.dtype, acc.x * inv); st_elem(out, at + 1, p.o.dtype, acc.y * inv);
    st_elem(out, at + 2, p.o.dtype, acc.z * inv); st_elem(out, at + 3, p.o.dtype, acc.w * inv);
}

void carve_workspace(DecodeParams& p, void* ws) {
    const size_t n = (size_t)p.B * p.n_chunks * p.Hq;
    const size_t npad = (n + 3) & ~(size_t)3;  // keeps the o partials 16-byte aligned
    p.ws_m = reinterpret_cast<float*>(ws);
    p.ws_l = p.ws_m + npad;
    p.ws_o = p.ws_l + npad;
}

// Partial results (chunks over all sequences) a call may produce: one per 128 positions, or, for small batches, whose chunks
// are cut finer, one per 32 as long as the scratch stays below kSmallScratch.  Grows with B and L, so that a buffer sized for the
// largest step serves every smaller one.
constexpr size_t kSmallScratch = (size_t)15 << 19;
// lisa_attn_shared_decode_static refuses a step whose scratch is larger than its array, so what finer chunks ask for has to fit with the
// padding of decode_workspace (the m and l arrays to whole float4, the whole to 256 bytes): no step of 128-position chunks that fits may be lost.
static_assert(kSmallScratch + 2 * 3 * sizeof(float) + 255 <= LISA_STATIC_SCRATCH_BYTES, "finer chunks must fit the scratch of the static call");
int64_t max_parts(int B, int Hq, int d, int L) {
    const int64_t coarse = (int64_t)B * ((L + kChunk - 1) / kChunk), fine = (int64_t)B * ((L + 31) / 32);
    if (d != 128) return coarse;
    return std::max(coarse, std::min(fine, (int64_t)(kSmallScratch / ((size_t)Hq * (d + 2) * sizeof(float)))));
}

bool vec16(const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; }

// Chunk length for a launch that runs `groups` CTAs per chunk: 128 once that gives every SM a CTA, else 64 or 32 (never more
// partial results than the workspace holds).
int chunk_length(int B, int Hq, int L, int64_t groups) {
    const int64_t want = sm_count(), most = max_parts(B, Hq, 128, L);
    int ch = kChunk;
    while (ch > 32 && B * (int64_t)((L + ch - 1) / ch) * groups < want && B * (int64_t)((L + ch / 2 - 1) / (ch / 2)) <= most) ch /= 2;
    return ch;
}
void set_chunk(DecodeParams& p, int ch, void* ws) {
    p.chunk = ch;
    p.n_chunks = (p.L_uniform + ch - 1) / ch;
    carve_workspace(p, ws);
}

// Two or three CTAs per SM: a CTA of the three-per-SM build takes about 1.3 times as long as one of the two-per-SM build runs
// beside one neighbour (B 64, L 4096, 40 heads: 0.510 against 0.528 ms for the whole grid), and the grid runs in whole waves of
// CTAs: take the build whose waves cost less.
bool three_per_sm(int64_t ctas) {
    const int64_t sms = sm_count();
    return 1.3 * (double)((ctas + 3 * sms - 1) / (3 * sms)) < (double)((ctas + 2 * sms - 1) / (2 * sms));
}

// Batches with given lengths whose grid is not resident at once have their chunks dealt to the CTAs (decode_item).  A smaller grid leaves an SM
// at most one CTA with work or two whichever way; there the count costs more than it gives (paper's default layer, 16 sequences of up to 1500:
// 70.5 us dealt, 66.8 not; 16 of up to 2900 of the 8B shape: an anchor and three layers 148 us dealt, 168 not; 16 of up to 3000, 40 heads: 80 and 92).
// A larger grid evens itself out (spread over [L / 8, L], 100 sequences of up to 1150, 900 CTAs: 306 us dealt, 289 not; 30 of up to 1900, 450 CTAs:
// 145 and 144) unless most sequences are short (four fifths at L / 8: 172 and 176, 125 and 133), and loses 1 to 5 % where they are all long.  With
// fewer than four chunks to the longest sequence nearly every CTA has positions (63 of up to 99, 40 heads, an anchor and three layers: 140 us dealt,
// 118 not).
bool deal_chunks(const DecodeParams& p, int64_t ctas) {
    const int64_t sms = sm_count();
    return p.seq_lens && p.B > 1 && p.B <= kDenseMaxB && p.n_chunks >= 4 && ctas > 2 * sms && ctas <= 3 * sms;
}

// KV heads whose V the CTAs of a grid that is resident at once ask into L2 behind their K or K' (k_row bytes a position and head); -1: the grid
// is not resident.  All of a chunk at once (paper's default model, 8 x 1111: 146 MB for the anchor layer, 85 for a shared one) stands in the
// queue for HBM before the score rows and K', and the anchor's is more than L2 holds; V is needed last: anchor and two shared layers
// 108.6 -> 102.8 us, the same with 24, 32, 36 and 48 MB, 107.5 with 110.  Small batches (1 x 333, 7B-shaped: 7 MB a layer) ask for all.
constexpr int64_t kPrefetchBytes = (int64_t)48 << 20;
int plan_prefetch(const DecodeParams& p, int64_t ctas, int n_kv, int k_row) {
    if (ctas > 2 * (int64_t)sm_count()) return -1;
    return (int)std::max<int64_t>(0, (kPrefetchBytes / (ctas * p.chunk) - (int64_t)n_kv * k_row) / 256);
}

template <int HQ, int HG, int CH, int M_C, int ENG>
cudaError_t launch_shared_fast(DecodeParams& p, cudaStream_t s) {
    const int64_t ctas = (int64_t)p.n_chunks * (HQ / HG) * p.B;
    const size_t smem = shared_fast_layout(HQ, HG, CH, ENG, p.m, HQ / p.Hkv).total;
    p.prefetch = plan_prefetch(p, ctas, HG / (HQ / p.Hkv), p.r * 2);
    auto launch = [&](auto kernel, dim3 grid) -> cudaError_t {
        const cudaError_t e = allow_smem(kernel, smem);
        return e != cudaSuccess ? e : launch_chained(kernel, grid, dim3(kDecodeThreads), smem, s, p);
    };
    const dim3 grid(p.n_chunks, HQ / HG, p.B);
    if constexpr (CH == 128) {   // (chunks are shorter only where the grid stays below deal_chunks' range, see chunk_length)
        const bool dealt = deal_chunks(p, ctas);
        p.least = 0;
        p.most = INT_MAX;
        if constexpr (ENG == kEngTf32) {
            const bool three = three_per_sm(ctas);
            if (three && !dealt) return launch(shared_decode_fast_kernel<HQ, HG, CH, M_C, ENG, 3, false>, grid);
            if (three) {
                // Which build suits a dealt batch depends on how many chunks hold positions, which only the device knows: both are launched, and
                // the one that the count is not for leaves at once.  Two CTAs per SM as long as that is one wave, three beyond (an anchor and three
                // shared layers, us, with both | two per SM alone | three alone | grid coordinates, lengths all alike and spread over [L / 8, L]:
                // 13 x 3079 with 8 KV heads 181 | 204 | 177 | 187 and 140 | 130 | 150 | 163; 12 x 3500 with 40 heads 453 | 520 | 440 | 454 and
                // 291 | 286 | 350 | 346).
                const int one_wave = 2 * sm_count() / (HQ / HG);
                p.least = one_wave + 1;
                const cudaError_t e = launch(shared_decode_fast_kernel<HQ, HG, CH, M_C, ENG, 3, true>, grid);
                if (e != cudaSuccess) return e;
                count_launches(1);
                p.least = 0;
                p.most = one_wave;
                return launch(shared_decode_fast_kernel<HQ, HG, CH, M_C, ENG, 2, true>, dim3(one_wave, HQ / HG));
            }
        }
        if (dealt) return launch(shared_decode_fast_kernel<HQ, HG, CH, M_C, ENG, 2, true>, grid);
    }
    return launch(shared_decode_fast_kernel<HQ, HG, CH, M_C, ENG, 2, false>, grid);
}

// The fast kernels' share of the shared layers; *taken says whether the call is one of them.
template <int HQ, int M_C>
cudaError_t shared_fast(DecodeParams& p, void* ws, cudaStream_t s, bool* taken) {
    const int G = p.Hq / p.Hkv;
    const bool bf16_w = p.w_dtype == LISA_BF16 && vec16(p.w1) && vec16(p.w2);
    const bool two = p.cache_dtype == LISA_BF16 && p.d == 128 && p.integrate != LISA_INTEGRATE_PLUS && p.ffn_layers == 2;
    const bool tf32 = two && p.integrate == LISA_INTEGRATE_ADD && p.m == M_C;
    *taken = tf32 || (two && bf16_w && p.m % 8 == 0);
    if (!*taken) return cudaSuccess;
    p.w_vec = bf16_w;
    const int64_t n_ctas = (int64_t)p.B * ((p.L_uniform + kChunk - 1) / kChunk), sms = sm_count();
    if (tf32) {
        // All heads to a CTA once that gives every SM two CTAs -- one with grouped queries, where the aligner is most of a CTA's work and
        // each group of heads would repeat half of it.  Else sixteen or eight heads to a CTA, then shorter chunks (7B-shaped, us:
        // B 64 L 300 55 -> 43 with 16 heads; B 8 L 1111 38 -> 25 with 8; B 4 L 1000 15.3 at 64 positions, 18.2 at 128).
        // CTAs are counted as if every sequence had L_uniform positions: the lengths of a ragged batch are on the device, where the host
        // cannot read them.  Spread over [L / 8, L], little more than half of the CTAs have positions, so such a batch gets longer chunks
        // than one of that size would.
        const int64_t want = G > 1 ? sms : 2 * sms;
        const bool full = 8 % G != 0 || n_ctas >= want;
        if (full) {
            set_chunk(p, kChunk, ws);
            return launch_shared_fast<HQ, HQ, 128, M_C, kEngTf32>(p, s);
        }
        if constexpr (HQ % 16 == 0)
            if (n_ctas * (HQ / 16) >= want) {
                set_chunk(p, kChunk, ws);
                return launch_shared_fast<HQ, 16, 128, M_C, kEngTf32>(p, s);
            }
        set_chunk(p, chunk_length(p.B, p.Hq, p.L_uniform, HQ / 8), ws);
        if (p.chunk == 128) return launch_shared_fast<HQ, 8, 128, M_C, kEngTf32>(p, s);
        if (p.chunk == 64) return launch_shared_fast<HQ, 8, 64, M_C, kEngTf32>(p, s);
        return launch_shared_fast<HQ, 8, 32, M_C, kEngTf32>(p, s);
    }
    set_chunk(p, chunk_length(p.B, p.Hq, p.L_uniform, 1), ws);
    if (p.integrate == LISA_INTEGRATE_ADD) {
        if (p.chunk == 128) return launch_shared_fast<HQ, HQ, 128, 0, kEngAdd>(p, s);
        if (p.chunk == 64) return launch_shared_fast<HQ, HQ, 64, 0, kEngAdd>(p, s);
        return launch_shared_fast<HQ, HQ, 32, 0, kEngAdd>(p, s);
    }
    if (p.chunk == 128) return launch_shared_fast<HQ, HQ, 128, 0, kEngConcat>(p, s);
    if (p.chunk == 64) return launch_shared_fast<HQ, HQ, 64, 0, kEngConcat>(p, s);
    return launch_shared_fast<HQ, HQ, 32, 0, kEngConcat>(p, s);
}

// Whether the merge lets its successor in behind its wait instead of at its start.  The kernels behind it ask their caches and weights into L2
// and stage the aligner when they start.  With few positions in the batch there is little to stream, and that early start only stands in the way of
// a chunk kernel that waits for its own loads; with more, or with merges enough to fill the SMs behind the chunks, it is worth its while.  An anchor
// and three layers, us, released early | late: one sequence of 640 positions 53.1 | 46.5 (7B-shaped), 52.6 | 48.4 (8B), 56.2 | 49.6 (13B), 78.0 | 72.2
// (paper's default), 5 x 200 54.0 | 50.6, 55.2 | 51.3, 55.6 | 55.1 and 88.4 | 86.9; beyond the lines 8 x 700 89.0 | 95.6 (7B), 20 x 700 102 | 112 (8B),
// 6 x 700 93.0 | 97.8 (13B), 1 x 2500 70.2 | 72.4 (7B), and 8 x 100 and 20 x 30 of the paper's default 72.9 | 81.2 and 83.5 | 87.2, although
// 20 x 30 of the others gains (53.9 | 49.5, 53.6 | 51.3, 56.1 | 53.7).
constexpr int kLatePositions = 1024;
bool merge_releases_late(const DecodeParams& p) {
    return (int64_t)p.B * p.L_uniform <= kLatePositions && 2 * (int64_t)p.Hq * p.B <= 3 * (int64_t)sm_count();
}

cudaError_t launch_merge(DecodeParams& p, cudaStream_t s) {
    p.late_release = merge_releases_late(p);
    const int each = kMergeThreads * 4 / p.d;   // chunks that the CTA's threads take side by side
    const int64_t ctas = (int64_t)p.Hq * p.B, sms = sm_count();
    auto kernel = p.n_chunks <= each || ctas > 10 * sms      ? decode_merge_kernel<1>
                  : p.n_chunks <= 2 * each || ctas > 8 * sms ? decode_merge_kernel<2>
                                                             : decode_merge_kernel<8>;
    const cudaError_t e = launch_chained(kernel, dim3(p.Hq, p.B), dim3(kMergeThreads), 0, s, p);
    count_launches(2);
    return e;
}

}  // namespace

// Dynamic shared memory of the general shared-layer chunk kernel: scores [Hq][kChunk], q' [Hq][kMaxRank], W1 and W2 (with
// some slack), b1, b2.
size_t shared_decode_smem(int Hq, int m_link, int integrate) {
    const int h_in = integrate == LISA_INTEGRATE_CONCAT ? 2 * Hq : Hq;
    const int m = integrate == LISA_INTEGRATE_PLUS ? 0 : m_link;
    return sizeof(float) * ((size_t)Hq * kChunk + (size_t)Hq * kMaxRank + (size_t)h_in * (m + 8) + (size_t)m * (Hq + 4) + m + Hq + 8);
}

size_t decode_workspace(int B, int Hq, int d, int L) {
    const size_t n = (size_t)max_parts(B, Hq, d, L) * Hq;
    const size_t npad = (n + 3) & ~(size_t)3;
    size_t bytes = (2 * npad + n * d) * sizeof(float);
    return (bytes + 255) & ~(size_t)255;
}

cudaError_t launch_shared_decode(const lisa_shared_decode_args& a, void* ws, cudaStream_t s) {
    const lisa_kvcache_layer& c = *a.cache;
    DecodeParams p{};
    p.B = a.B; p.Hq = a.Hq; p.Hkv = c.Hkv; p.d = c.d; p.L_cap = c.L_cap; p.L_uniform = a.L;
    p.seq_lens = a.seq_lens;
    p.prev = a.prev_scores; p.prev_sb = a.prev_stride_b; p.prev_sh = a.prev_stride_h;
    p.qp = make_view(a.link.qp);
    p.kpT = c.k; p.vcache = c.v; p.cache_dtype = c.dtype;
    p.r = c.r; p.m = a.link.m; p.act = a.link.act; p.integrate = a.link.integrate; p.ffn_layers = a.link.ffn_layers;
    p.w_dtype = a.link.w_dtype;
    p.w1 = a.link.w1; p.b1 = a.link.b1; p.w2 = a.link.w2; p.b2 = a.link.b2;
    p.out_scores = a.out_scores; p.sc_sb = a.scores_stride_b; p.sc_sh = a.scores_stride_h;
    p.row_bf16 = a.scores_dtype == LISA_BF16;
    p.o = make_view(a.o);
    cudaError_t e = cudaSuccess;
    bool taken = false;
    if (p.Hq == 40) e = shared_fast<40, 80>(p, ws, s, &taken);
    else if (p.Hq == 32) e = shared_fast<32, 64>(p, ws, s, &taken);
    if (!taken) {
        set_chunk(p, kChunk, ws);
        const size_t smem = shared_decode_smem(p.Hq, p.m, p.integrate);
        auto kernel = p.row_bf16 ? shared_decode_chunk_kernel<true> : shared_decode_chunk_kernel<false>;
        if ((e = allow_smem(kernel, smem)) != cudaSuccess) return e;
        e = launch_chained(kernel, dim3(p.n_chunks, p.B), dim3(kThreads), smem, s, p);
    }
    return e == cudaSuccess ? launch_merge(p, s) : e;
}

cudaError_t launch_anchor_decode(const lisa_anchor_args& a, void* ws, cudaStream_t s) {
    const lisa_kvcache_layer& c = *a.cache;
    DecodeParams p{};
    p.B = a.B; p.Hq = a.Hq; p.Hkv = c.Hkv; p.d = c.d; p.L_cap = c.L_cap; p.L_uniform = a.L;
    p.seq_lens = a.seq_lens;
    p.q = make_view(a.q);
    p.kcache = c.k; p.vcache = c.v; p.cache_dtype = c.dtype;
    p.out_scores = a.out_scores; p.sc_sb = a.scores_stride_b; p.sc_sh = a.scores_stride_h;
    p.row_bf16 = a.scores_dtype == LISA_BF16;
    p.o = make_view(a.o);
    const int G = p.Hq / p.Hkv;
    const TView& q = p.q;
    cudaError_t e;
    if (p.cache_dtype == LISA_BF16 && p.d == 128 && q.dtype == LISA_BF16 && vec16(q.ptr) && q.sb % 8 == 0 && q.sh % 8 == 0) {
        // Eight KV heads to a CTA, one per warp: CTAs small enough for even waves, nothing computed twice (40 heads, us: B 12 L 3500
        // 178 -> 138 against all heads to a CTA, B 64 L 4096 803 -> 790).  Fewer, then shorter chunks, where that does not give
        // every SM a CTA (counted as in shared_fast, ragged batches as if they were uniform).
        const int64_t want = sm_count(), chunks = (int64_t)p.B * ((a.L + kChunk - 1) / kChunk);
        int kv = std::min(8, p.Hkv);
        while (p.Hkv % kv) --kv;
        while (kv % 2 == 0 && chunks * (p.Hkv / kv) < want) kv /= 2;
        p.heads = kv * G;
        set_chunk(p, chunk_length(p.B, p.Hq, a.L, p.Hkv / kv), ws);
        const int64_t ctas = (int64_t)p.n_chunks * p.B * (p.Hkv / kv);
        p.prefetch = plan_prefetch(p, ctas, kv, 256);
        const bool dealt = deal_chunks(p, ctas);   // (only with whole chunks, see launch_shared_fast)
        p.least = 0;
        p.most = INT_MAX;
        const size_t smem = anchor_fast_smem(p.heads, p.chunk, G);
        auto kernel = dealt          ? anchor_decode_fast_kernel<128, true>
                      : p.chunk == 128 ? anchor_decode_fast_kernel<128, false>
                      : p.chunk == 64  ? anchor_decode_fast_kernel<64, false>
                                       : anchor_decode_fast_kernel<32, false>;
        if ((e = allow_smem(kernel, smem)) != cudaSuccess) return e;
        e = launch_chained(kernel, dim3(p.n_chunks, p.Hkv / kv, p.B), dim3(kDecodeThreads), smem, s, p);
    } else {
        set_chunk(p, kChunk, ws);
        const size_t smem = sizeof(float) * ((size_t)p.Hq * kChunk + (size_t)p.Hq * p.d);
        if ((e = allow_smem(anchor_decode_chunk_kernel, smem)) != cudaSuccess) return e;
        e = launch_chained(anchor_decode_chunk_kernel, dim3(p.n_chunks, p.B), dim3(kThreads), smem, s, p);
    }
    return e == cudaSuccess ? launch_merge(p, s) : e;
}

}  // namespace lisa
