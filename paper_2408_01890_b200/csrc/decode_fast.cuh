// Decode kernels for bf16 caches of head width 128 (decode.cu holds the general ones and the dispatch).
//
// A CTA takes CH cached positions of one sequence and HG of its query heads.  CH = 128 and all heads read everything once and
// are right once there are CTAs enough; with few sequences or short contexts such a grid leaves most SMs idle (one
// sequence of 333 positions: three CTAs, 38 us a layer), so positions are cut finer (64, 32: more partial results for the merge,
// nothing computed twice) and the heads are divided as well (the first FFN layer, which every head needs, is then computed by
// each group again).  All 8 warps work in every phase whatever CH is: with fewer than 8 strips of 16 positions the FFN's
// hidden units are divided over HS = 128 / CH warps per strip and their partial sums added in a fixed order.
// K and V rows are read once for all query heads of a group of up to four (GV) that share them.  Where the sequence ends inside a chunk,
// rows past its end count as zeros, with probability zero (any other stand-in would turn into NaN where it holds an infinity), so that
// every chunk runs the pipelined code (a loop with one row in flight took 120 us over a last chunk).
#pragma once
#include <type_traits>

#include "decode_common.cuh"

namespace lisa {

constexpr int kEngTf32 = 0;    // ADD, two-layer FFN of compile-time width: tf32 operands (scores rounded to 11 bits)
constexpr int kEngAdd = 1;     // ADD, two-layer FFN of any width up to 256: fp32 operands as three bf16 terms, bf16 weights
constexpr int kEngConcat = 2;  // the same with the difference as second half of the input

// Query heads that share a pass over the rows of their KV head.
__host__ __device__ inline int kv_group(int G) { return G % 4 == 0 ? 4 : G % 2 == 0 ? 2 : 1; }
// 16-byte loads per lane in one of the two register sets of a streaming warp (two rows per load and warp): with four heads the
// accumulators take the registers of the other half.
__host__ __device__ constexpr int stream_loads(int gv) { return gv == 4 ? 4 : 8; }
// Ranges a chunk's rows are cut into where a CTA has fewer KV heads than warps.
__host__ __device__ inline int row_parts(int nv, int ch, int gv) {
    const int a = nv >= kDecodeWarps ? 1 : kDecodeWarps / nv, b = ch / (2 * stream_loads(gv));
    return a < b ? a : b;
}

// Where a work item's rows start: `base` is row 0 of the chunk in KV head 0 of the CTA's group, heads lie head_stride
// 16-byte units apart, a row is 16 units; the chunk has nrows valid rows.
struct Rows {
    const uint4* base;
    size_t head_stride;
    int nrows;
};

// Streams the rows of nv virtual KV heads (vper of them on each KV head) through body(regs, v, row0): one warp per head, or per (head,
// range of rows); two register sets of U 16-byte loads per lane alternate, across heads too.  A lane holds the 16 bytes `lane % 16` of
// rows row0 + 2 u + lane / 16.  done(v, part) is called behind a head's (or range's) last body.
template <int CH, int U, typename Body, typename Done>
__device__ __forceinline__ void stream_rows(const Rows& r, int nv, int vper, int ps, Body body, Done done) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane & 15, rsel = lane >> 4;
    constexpr int ROWS = 2 * U, NB = CH / ROWS;
    if (r.nrows == CH && ps == 1) {   // a full chunk: every offset a compile-time constant off one pointer
        if (warp >= nv) return;
        auto head_ptr = [&](int v) { return r.base + (size_t)(v / vper) * r.head_stride + rsel * 16 + sub; };
        auto load = [&](uint4* q, const uint4* hp, int bt) {
#pragma unroll
            for (int u = 0; u < U; ++u) q[u] = ld_stream16(hp + (bt * ROWS + 2 * u) * 16);
        };
        const uint4* hp = head_ptr(warp);
        uint4 qa[U], qb[U];
        load(qa, hp, 0);
        for (int v = warp; v < nv; v += kDecodeWarps) {
            const bool has_next = v + kDecodeWarps < nv;
            const uint4* np = has_next ? head_ptr(v + kDecodeWarps) : hp;
            // (groups of four heads: the unrolled code would not stay in the instruction cache, 188 instead of 184 us at B 32, L 8192)
#pragma unroll(U == 8 ? NB / 2 : 1)
            for (int bt = 0; bt < NB; bt += 2) {
                load(qb, hp, bt + 1);
                body(qa, v, bt * ROWS);
                if (bt + 2 < NB) load(qa, hp, bt + 2);
                else if (has_next) load(qa, np, 0);
                body(qb, v, (bt + 1) * ROWS);
            }
            done(v, 0);
            hp = np;
        }
        return;
    }
    const int part = warp / nv * (ps > 1), first = ps > 1 ? warp % nv : warp;
    if (first >= nv || part >= ps) return;
    const int nb_all = (r.nrows + ROWS - 1) / ROWS, b0 = nb_all * part / ps, b1 = nb_all * (part + 1) / ps;
    if (b0 == b1) return;
    auto load = [&](uint4* q, int v, int bt) {
        const uint4* p = r.base + (size_t)(v / vper) * r.head_stride + (bt * ROWS + rsel) * 16 + sub;
        const int left = r.nrows - bt * ROWS - rsel;
#pragma unroll
        for (int u = 0; u < U; ++u) q[u] = ld_stream16_or_zero(p + u * 32, 2 * u < left);
    };
    uint4 qa[U], qb[U];
    int lv = first, lb = b0;      // next batch to load
    auto load_next = [&](uint4* q) {
        if (lv < nv) {
            load(q, lv, lb);
            if (++lb == b1) { lb = b0; lv += ps > 1 ? nv : kDecodeWarps; }
        }
    };
    load_next(qa);
    int v = first, bt = b0;
    while (true) {
        load_next(qb);
        body(qa, v, bt * ROWS);
        if (++bt == b1) { done(v, part); bt = b0; v += ps > 1 ? nv : kDecodeWarps; if (v >= nv) break; }
        load_next(qa);
        body(qb, v, bt * ROWS);
        if (++bt == b1) { done(v, part); bt = b0; v += ps > 1 ? nv : kDecodeWarps; if (v >= nv) break; }
    }
}

// Partial P.V of a chunk: s_s[head][ld] holds the exponentials (zero past the sequence's end), red scratch for position ranges beyond
// the first ((ps - 1) x HG x 128 floats); results go to out[head][128].
template <int CH, int GV>
__device__ __forceinline__ void pv_stream(const Rows& r, int nv, int vper, const float* s_s, int ld, float* red, float* out) {
    constexpr int U = stream_loads(GV);
    const int lane = threadIdx.x & 31, sub = lane & 15, rsel = lane >> 4, ps = row_parts(nv, CH, GV);
    float acc[GV][8];
#pragma unroll
    for (int q = 0; q < GV; ++q)
#pragma unroll
        for (int t = 0; t < 8; ++t) acc[q][t] = 0.f;
    auto body = [&](const uint4* regs, int v, int row0) {
        const float* ps_ = s_s + v * GV * ld + row0 + rsel;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float f[8];
            bf16x8_to_f32(regs[u], f);
#pragma unroll
            for (int q = 0; q < GV; ++q) {
                const float pj = ps_[q * ld + 2 * u];
#pragma unroll
                for (int t = 0; t < 8; ++t) acc[q][t] = fmaf(pj, f[t], acc[q][t]);
            }
        }
    };
    auto done = [&](int v, int part) {
#pragma unroll
        for (int q = 0; q < GV; ++q) {
#pragma unroll
            for (int t = 0; t < 8; ++t) acc[q][t] += __shfl_xor_sync(0xffffffffu, acc[q][t], 16);
            if (rsel == 0) {
                float4* dst = reinterpret_cast<float4*>((part == 0 ? out : red + (size_t)(part - 1) * nv * GV * 128) + (size_t)(v * GV + q) * 128 + sub * 8);
                dst[0] = make_float4(acc[q][0], acc[q][1], acc[q][2], acc[q][3]);
                dst[1] = make_float4(acc[q][4], acc[q][5], acc[q][6], acc[q][7]);
            }
#pragma unroll
            for (int t = 0; t < 8; ++t) acc[q][t] = 0.f;
        }
    };
    stream_rows<CH, U>(r, nv, vper, ps, body, done);
    if (ps > 1) {   // add the ranges, in order; a range without rows wrote nothing
        __syncthreads();
        const int nb = (r.nrows + 2 * U - 1) / (2 * U);
        for (int e = threadIdx.x; e < nv * GV * 32; e += kDecodeThreads) {
            float4 v = nb / ps > 0 ? reinterpret_cast<float4*>(out)[e] : make_float4(0.f, 0.f, 0.f, 0.f);
            for (int q = 1; q < ps; ++q) {
                if (nb * (q + 1) / ps == nb * q / ps) continue;
                const float4 x = reinterpret_cast<const float4*>(red + (size_t)(q - 1) * nv * GV * 128)[e];
                v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
            }
            reinterpret_cast<float4*>(out)[e] = v;
        }
    }
}

// Scores of a chunk: s_s[head][j] = scale * q_head . K_j; q_s [head][128] fp32.  A lane holds the partial dot products of U rows and GV
// heads over its 8 of the 128 dimensions; the sum over the 16 lanes of a row is a butterfly that halves the number of live values
// at every step.
template <int CH, int GV>
__device__ __forceinline__ void qk_stream(const Rows& r, int nv, int vper, const float* q_s, float* s_s, int ld, float scale) {
    constexpr int U = stream_loads(GV), NV = GV * U;   // 8 or 16 values
    const int lane = threadIdx.x & 31, sub = lane & 15, rsel = lane >> 4;
    auto body = [&](const uint4* regs, int v, int row0) {
        float dot[NV];
#pragma unroll
        for (int q = 0; q < GV; ++q) {
            const float4* qp = reinterpret_cast<const float4*>(q_s + (v * GV + q) * 128 + sub * 8);
            const float4 a = qp[0], b = qp[1];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float f[8];
                bf16x8_to_f32(regs[u], f);
                float s = a.x * f[0];
                s = fmaf(a.y, f[1], s); s = fmaf(a.z, f[2], s); s = fmaf(a.w, f[3], s);
                s = fmaf(b.x, f[4], s); s = fmaf(b.y, f[5], s); s = fmaf(b.z, f[6], s);
                dot[q * U + u] = fmaf(b.w, f[7], s);
            }
        }
        int n = NV / 2;
#pragma unroll
        for (int bit = 8; bit >= 16 / NV; bit >>= 1, n >>= 1) {
#pragma unroll
            for (int i = 0; i < NV / 2; ++i)
                if (i < n) {
                    const float send = (sub & bit) ? dot[i] : dot[i + n];
                    const float keep = (sub & bit) ? dot[i + n] : dot[i];
                    dot[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
                }
        }
        int idx = sub;   // the value this lane ends up with: q * U + u
        if constexpr (NV == 8) {
            dot[0] += __shfl_xor_sync(0xffffffffu, dot[0], 1);
            idx = sub >> 1;
        }
        if (NV == 16 || (sub & 1) == 0) s_s[(v * GV + idx / U) * ld + row0 + 2 * (idx % U) + rsel] = dot[0] * scale;
    };
    stream_rows<CH, U>(r, nv, vper, row_parts(nv, CH, GV), body, [](int, int) {});
}

// Softmax of a chunk per head, in place: s_s[head][CH] scores (add_s), plus HS partial sums y_s[hs][head][CH] where y_s is given,
// become exponentials; the finished scores go to the row of the next layer, maximum and sum to the workspace.
template <int CH, int HS>
__device__ __forceinline__ void finish_scores(const DecodeParams& p, float* s_s, const float* y_s, bool add_s, int HG, int h0, int b, int j0, int nrows, size_t part) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int PL = CH / 32;
    for (int h = warp; h < HG; h += kDecodeWarps) {
        float v[PL], cmax = -INFINITY;
        const int64_t row = b * p.sc_sb + (h0 + h) * p.sc_sh + j0;
#pragma unroll
        for (int t = 0; t < PL; ++t) {
            const int pos = lane + 32 * t;
            float x = add_s ? s_s[h * CH + pos] : 0.f;
            if (y_s) {
#pragma unroll
                for (int q = 0; q < HS; ++q) x += y_s[(q * HG + h) * CH + pos];
            }
            if (pos < nrows) {
                if (p.out_scores) {
                    if (p.row_bf16) st_row<true>(p.out_scores, row + pos, x);
                    else st_row<false>(p.out_scores, row + pos, x);
                }
            } else {
                x = -INFINITY;
            }
            v[t] = x;
            cmax = fmaxf(cmax, x);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, off));
        float sum = 0.f;
#pragma unroll
        for (int t = 0; t < PL; ++t) {
            const float e = __expf(v[t] - cmax);
            s_s[h * CH + lane + 32 * t] = e;
            sum += e;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
        if (lane == 0) {
            p.ws_m[part + h] = cmax;
            p.ws_l[part + h] = sum;
        }
    }
}

template <int CH>
__device__ __forceinline__ void pv_chunk(const DecodeParams& p, const float* s_s, float* red, int b, int kv0, int HG, int j0, int nrows, float* out) {
    const int G = p.Hq / p.Hkv, gv = kv_group(G);
    const Rows rows{reinterpret_cast<const uint4*>(p.vcache) + (((size_t)b * p.Hkv + kv0) * p.L_cap + j0) * 16, (size_t)p.L_cap * 16, nrows};
    if (gv == 1) pv_stream<CH, 1>(rows, HG, G, s_s, CH, red, out);
    else if (gv == 2) pv_stream<CH, 2>(rows, HG / 2, G / 2, s_s, CH, red, out);
    else pv_stream<CH, 4>(rows, HG / 4, G / 4, s_s, CH, red, out);
}

// The caches of this CTA's chunk on their way into L2, before the wait for the preceding kernel: a hint (the length may be read before
// an earlier kernel has set it), and L2 is the point of coherence, so a new token's row that is still being written is read right later.
__device__ __forceinline__ void prefetch_chunk(const DecodeParams& p, int kv0, int n_kv, int ch, bool standard) {
    const int b = blockIdx.z, j0 = blockIdx.x * ch, hint = min(decode_length(p, b), p.L_cap) - j0;
    if (hint <= 0 || p.prefetch < 0) return;
    const int nrows = min(ch, hint), tid = threadIdx.x;
    const size_t row0 = ((size_t)b * p.Hkv + kv0) * p.L_cap + j0;
    auto bulk = [](const void* q, uint32_t bytes) { asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(q), "r"(bytes) : "memory"); };
    if (standard) {
        if (tid < n_kv) bulk(reinterpret_cast<const uint4*>(p.kcache) + (row0 + (size_t)tid * p.L_cap) * 16, nrows * 256);
    } else {
        const __nv_bfloat16* base = reinterpret_cast<const __nv_bfloat16*>(p.kpT) + ((size_t)b * p.Hkv + kv0) * p.r * p.L_cap + j0;
        const int lines = (nrows + 63) / 64;
        for (int e = tid; e < n_kv * p.r * lines; e += kDecodeThreads)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(base + (size_t)(e / lines) * p.L_cap + e % lines * 64) : "memory");
    }
    if (tid < min(n_kv, p.prefetch)) bulk(reinterpret_cast<const uint4*>(p.vcache) + (row0 + (size_t)tid * p.L_cap) * 16, nrows * 256);
}

// ---------------------------------------------------------------------------------------------
// Standard layer.  Shared memory: scores [HG][CH], queries fp32 [HG][128], position ranges of P.V.
// ---------------------------------------------------------------------------------------------
inline size_t anchor_fast_smem(int HG, int ch, int G) {
    const int gv = kv_group(G);
    return sizeof(float) * ((size_t)HG * ch + (size_t)row_parts(HG / gv, ch, gv) * HG * 128);
}

template <int CH, bool DENSE>
__global__ void __launch_bounds__(kDecodeThreads, 2) anchor_decode_fast_kernel(const __grid_constant__ DecodeParams p) {
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x;
    const int HG = p.heads, h0 = blockIdx.y * HG, G = p.Hq / p.Hkv, kv0 = h0 / G, gv = kv_group(G);
    chain_release();
    if constexpr (!DENSE) prefetch_chunk(p, kv0, HG / G, CH, true);
    chain_wait();
    int b, chunk, L;
    if (!decode_item<CH, DENSE>(p, b, chunk, L)) return;
    const int j0 = chunk * CH, nrows = min(CH, L - j0);
    float* s_s = smem;
    float* q_s = s_s + HG * CH;
    float* red = q_s + HG * 128;
    for (int e = tid; e < HG * 16; e += kDecodeThreads) {
        const int h = e >> 4, x = e & 15;
        float f[8];
        bf16x8_to_f32(*reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.q.ptr) + b * p.q.sb + (h0 + h) * p.q.sh + x * 8), f);
        float4* dst = reinterpret_cast<float4*>(q_s + h * 128 + x * 8);
        dst[0] = make_float4(f[0], f[1], f[2], f[3]);
        dst[1] = make_float4(f[4], f[5], f[6], f[7]);
    }
    __syncthreads();
    const Rows rows{reinterpret_cast<const uint4*>(p.kcache) + (((size_t)b * p.Hkv + kv0) * p.L_cap + j0) * 16, (size_t)p.L_cap * 16, nrows};
    const float scale = rsqrtf(128.f);
    if (gv == 1) qk_stream<CH, 1>(rows, HG, G, q_s, s_s, CH, scale);
    else if (gv == 2) qk_stream<CH, 2>(rows, HG / 2, G / 2, q_s, s_s, CH, scale);
    else qk_stream<CH, 4>(rows, HG / 4, G / 4, q_s, s_s, CH, scale);
    __syncthreads();
    const size_t part = ((size_t)b * p.n_chunks + chunk) * p.Hq + h0;
    finish_scores<CH, 1>(p, s_s, nullptr, true, HG, h0, b, j0, nrows, part);
    __syncthreads();
    pv_chunk<CH>(p, s_s, red, b, kv0, HG, j0, nrows, p.ws_o + part * 128);
}

// ---------------------------------------------------------------------------------------------
// Shared layer.
// ---------------------------------------------------------------------------------------------
// A_Delta of the chunk (Eq. 3): a warp takes a virtual KV head of GV query heads, a lane 8 positions and every RS-th rank row.
template <int CH, int GV>
__device__ __forceinline__ void delta_chunk(const DecodeParams& p, float* s_s, const float* qp_s, int b, int kv0, int HG, int j0) {
    constexpr int P8 = CH / 8, RS = 32 / P8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, j8 = lane % P8, rs = lane / P8;
    const int r = p.r, nv = HG / GV, vper = p.Hq / p.Hkv / GV;
    const bool in = j0 + j8 * 8 < p.L_cap;
    const float inv_sqrt_r = rsqrtf((float)r);
    for (int v = warp; v < nv; v += kDecodeWarps) {
        float acc[GV][8];
#pragma unroll
        for (int q = 0; q < GV; ++q)
#pragma unroll
            for (int t = 0; t < 8; ++t) acc[q][t] = 0.f;
        const __nv_bfloat16* base = reinterpret_cast<const __nv_bfloat16*>(p.kpT) + ((size_t)b * p.Hkv + kv0 + v / vper) * r * p.L_cap + j0 + j8 * 8;
        for (int x0 = rs; x0 < r; x0 += 8 * RS) {
            uint4 raw[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                raw[e] = in && x0 + e * RS < r ? ld_stream16(base + (size_t)(x0 + e * RS) * p.L_cap) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int x = x0 + e * RS < r ? x0 + e * RS : 0;   // (the loaded values are zero then)
                float f[8];
                bf16x8_to_f32(raw[e], f);
#pragma unroll
                for (int q = 0; q < GV; ++q) {
                    const float qx = qp_s[(v * GV + q) * kMaxRank + x];
#pragma unroll
                    for (int t = 0; t < 8; ++t) acc[q][t] = fmaf(qx, f[t], acc[q][t]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < GV; ++q) {
#pragma unroll
            for (int t = 0; t < 8; ++t) {
#pragma unroll
                for (int off = P8; off < 32; off <<= 1) acc[q][t] += __shfl_xor_sync(0xffffffffu, acc[q][t], off);
                acc[q][t] *= inv_sqrt_r;
            }
            if (rs == 0) {
                float4* dst = reinterpret_cast<float4*>(s_s + (v * GV + q) * CH + j8 * 8);
                dst[0] = make_float4(acc[q][0], acc[q][1], acc[q][2], acc[q][3]);
                dst[1] = make_float4(acc[q][4], acc[q][5], acc[q][6], acc[q][7]);
            }
        }
    }
}

__device__ __forceinline__ uint32_t to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}
// d += a (16x8, row) . b (8x8, col), tf32 in, fp32 accumulate
__device__ __forceinline__ void mma_tf32(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// d += a (16x16, row) . b (16x8, col), bf16 in, fp32 accumulate
__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t* r, const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
__device__ __forceinline__ void ldsm_x2_trans(uint32_t* r, const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1]) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}
// Two fp32 values as three packed bf16 pairs that add up to them (24 mantissa bits in three times 8).  The first term's rounding saturates:
// otherwise it would take the largest finite scores, a mask's for instance, to infinity.
__device__ __forceinline__ void split3(float x, float y, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(y), "f"(x));
    x -= __uint_as_float(hi << 16); y -= __uint_as_float(hi & 0xffff0000u);
    mid = pack2(x, y);
    x -= __uint_as_float(mid << 16); y -= __uint_as_float(mid & 0xffff0000u);
    lo = pack2(x, y);
}

// Shared memory of a CTA, in order (byte offsets): scores [HG][CH]; partial FFN outputs [HS][HG][CH] (HS > 1, and the concatenating
// form, whose scores stay the FFN's input); q' [HG][kMaxRank]; weights; b1, b2.  The position ranges of P.V go over the weights.
struct SharedFastLayout {
    size_t y, qp, w1, w2, b1, b2, total;
};
__host__ __device__ inline SharedFastLayout shared_fast_layout(int HQ, int HG, int CH, int eng, int m, int G) {
    SharedFastLayout l;
    const int HS = 128 / CH, mp = (m + 15) / 16 * 16, gv = kv_group(G);
    size_t off = (size_t)HG * CH * 4;
    l.y = off; off += (HS > 1 || eng == kEngConcat) ? (size_t)HS * HG * CH * 4 : 0;
    l.qp = off; off += (size_t)HG * kMaxRank * 4;
    l.w1 = off;
    if (eng == kEngTf32) {
        off += (size_t)HQ * (m + 8) * 4; l.w2 = off; off += (size_t)m * (HG + 4) * 4;
        l.b1 = off; off += (size_t)m * 4;
    } else {
        const int kp = eng == kEngConcat ? 2 * HQ : (HQ + 15) / 16 * 16;
        off += (size_t)kp * (mp + 8) * 2; l.w2 = off; off += (size_t)mp * (HG + 8) * 2;
        l.b1 = off; off += (size_t)mp * 4;
    }
    l.b2 = off; off += (size_t)HG * 4;
    const size_t red = l.w1 + (size_t)(row_parts(HG / gv, CH, gv) - 1) * HG * 128 * 4;
    l.total = off > red ? off : red;
    return l;
}

// CTAS: CTAs per SM the kernel is compiled for.  Three hide the FFN phase (no loads in flight from the CTA that is in it) better than
// two, at 80 instead of 128 registers; which one a launch takes depends on how its grid fills the waves.
template <int HQ, int HG, int CH, int M_C, int ENG, int CTAS, bool DENSE>
__global__ void __launch_bounds__(kDecodeThreads, CTAS) shared_decode_fast_kernel(const __grid_constant__ DecodeParams p) {
    static_assert(ENG == kEngTf32 ? M_C > 0 : HG == HQ, "the split forms run with all heads");
    constexpr int HS = 128 / CH, NT2 = HG / 8;
    extern __shared__ __align__(16) uint8_t smem_b[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int h0 = blockIdx.y * HG, G = HQ / p.Hkv, kv0 = h0 / G;
    const int m = ENG == kEngTf32 ? M_C : p.m;
    chain_release();
    if constexpr (!DENSE) prefetch_chunk(p, kv0, HG / G, CH, false);
    const SharedFastLayout lay = shared_fast_layout(HQ, HG, CH, ENG, m, G);
    float* s_s = reinterpret_cast<float*>(smem_b);
    float* y_s = reinterpret_cast<float*>(smem_b + lay.y);
    float* qp_s = reinterpret_cast<float*>(smem_b + lay.qp);
    float* b1_s = reinterpret_cast<float*>(smem_b + lay.b1);
    float* b2_s = reinterpret_cast<float*>(smem_b + lay.b2);

    // the aligner's weights are constants of the model: staged while the kernel before this one may still be running
    const int mp = (m + 15) / 16 * 16;
    if constexpr (ENG == kEngTf32) {   // rows [HQ][M + 8], [M][HG + 4]: padded so that fragment loads spread over the banks
        float* w1_s = reinterpret_cast<float*>(smem_b + lay.w1);
        float* w2_s = reinterpret_cast<float*>(smem_b + lay.w2);
        if (p.w_vec) {
            auto put = [](float* dst, const uint4& v) {
                float f[8];
                bf16x8_to_f32(v, f);
                float4* d = reinterpret_cast<float4*>(dst);
                d[0] = make_float4(f[0], f[1], f[2], f[3]);
                d[1] = make_float4(f[4], f[5], f[6], f[7]);
            };
            const __nv_bfloat16 *g1 = reinterpret_cast<const __nv_bfloat16*>(p.w1), *g2 = reinterpret_cast<const __nv_bfloat16*>(p.w2);
            for (int e = tid; e < HQ * (M_C / 8); e += kDecodeThreads) {
                const int k = e / (M_C / 8), c = e % (M_C / 8) * 8;
                put(w1_s + k * (M_C + 8) + c, *reinterpret_cast<const uint4*>(g1 + k * M_C + c));
            }
            for (int e = tid; e < M_C * NT2; e += kDecodeThreads) {
                const int k = e / NT2, c = e % NT2 * 8;
                put(w2_s + k * (HG + 4) + c, *reinterpret_cast<const uint4*>(g2 + k * HQ + h0 + c));
            }
        } else {
            for (int e = tid; e < HQ * M_C; e += kDecodeThreads) w1_s[(e / M_C) * (M_C + 8) + e % M_C] = ld_elem(p.w1, e, p.w_dtype);
            for (int e = tid; e < M_C * HG; e += kDecodeThreads) w2_s[(e / HG) * (HG + 4) + e % HG] = ld_elem(p.w2, (e / HG) * HQ + h0 + e % HG, p.w_dtype);
        }
    } else {   // bf16 weights as they are, zero rows and columns beyond the FFN's sizes
        __nv_bfloat16* w1_s = reinterpret_cast<__nv_bfloat16*>(smem_b + lay.w1);   // [inputs][mp + 8]
        __nv_bfloat16* w2_s = reinterpret_cast<__nv_bfloat16*>(smem_b + lay.w2);   // [mp][HG + 8]
        constexpr int H_IN = ENG == kEngConcat ? 2 * HQ : HQ, KP = ENG == kEngConcat ? 2 * HQ : (HQ + 15) / 16 * 16;
        const int c8 = mp / 8;
        for (int e = tid; e < KP * c8; e += kDecodeThreads) {
            const int k = e / c8, c = (e - k * c8) * 8;
            *reinterpret_cast<uint4*>(w1_s + k * (mp + 8) + c) =
                k < H_IN && c < m ? *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.w1) + k * m + c) : make_uint4(0u, 0u, 0u, 0u);
        }
        for (int e = tid; e < mp * NT2; e += kDecodeThreads) {
            const int k = e / NT2, c = e % NT2 * 8;
            *reinterpret_cast<uint4*>(w2_s + k * (HG + 8) + c) =
                k < m ? *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.w2) + k * HQ + c) : make_uint4(0u, 0u, 0u, 0u);
        }
    }
    for (int e = tid; e < (ENG == kEngTf32 ? m : mp); e += kDecodeThreads) b1_s[e] = e < m ? ldw(p.b1, e, p.w_dtype) : 0.f;
    for (int e = tid; e < HG; e += kDecodeThreads) b2_s[e] = ldw(p.b2, h0 + e, p.w_dtype);
    chain_wait();   // from here on: lengths, Q', the caches and the score row, which earlier kernels of the stream produce
    int b, chunk, L;
    if (!decode_item<CH, DENSE>(p, b, chunk, L)) return;
    const int j0 = chunk * CH, nrows = min(CH, L - j0);
    {   // at most HG * kMaxRank values: all loads in flight together
        constexpr int NQ = HG * kMaxRank / kDecodeThreads;
        auto fetch = [&](const auto* q) {
            q += b * p.qp.sb + h0 * p.qp.sh;
            float v[NQ];
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                const int e = tid + i * kDecodeThreads, h = e / kMaxRank, x = e % kMaxRank;
                v[i] = x < p.r ? (float)q[h * p.qp.sh + x] : 0.f;
            }
#pragma unroll
            for (int i = 0; i < NQ; ++i) qp_s[tid + i * kDecodeThreads] = v[i];
        };
        if (p.qp.dtype == LISA_BF16) fetch(reinterpret_cast<const __nv_bfloat16*>(p.qp.ptr));
        else fetch(reinterpret_cast<const float*>(p.qp.ptr));
    }
    __syncthreads();
    {
        const int gv = kv_group(G);
        if (gv == 1) delta_chunk<CH, 1>(p, s_s, qp_s, b, kv0, HG, j0);
        else if (gv == 2) delta_chunk<CH, 2>(p, s_s, qp_s, b, kv0, HG, j0);
        else delta_chunk<CH, 4>(p, s_s, qp_s, b, kv0, HG, j0);
    }
    if constexpr (HS == 1 || ENG == kEngConcat) __syncthreads();

    // ---- the aligner's FFN: a warp owns 16 positions (M dimension) and every HS-th slice of hidden units ----
    const int g = lane >> 2, t = lane & 3;
    const int strip = warp % (CH / 16), hs = warp / (CH / 16);
    const int p0 = strip * 16 + g, p1 = p0 + 8;             // this lane's two position rows
    const bool ok0 = p0 < nrows, ok1 = p1 < nrows;
    // every score this lane feeds to the first layer, all loads in flight together; slots come in pairs that start at heads 0, 8, ...
    constexpr int NPREV = ENG == kEngTf32 ? HQ / 4 : (HQ + 15) / 16 * 4;
    float pv[NPREV][2];
    auto load_prev = [&](auto* row) {
        row += b * p.prev_sb + j0 + (ENG == kEngTf32 ? t : 2 * t) * p.prev_sh;
        const int64_t s1 = (ENG == kEngTf32 ? 4 : 1) * p.prev_sh, s8 = 8 * p.prev_sh;
#pragma unroll
        for (int k = 0; k < NPREV; k += 2, row += s8) {
            const bool in = HQ % 16 == 0 || ENG == kEngTf32 || k < HQ / 4;
            pv[k][0] = in && ok0 ? (float)row[p0] : 0.f;
            pv[k][1] = in && ok1 ? (float)row[p1] : 0.f;
            pv[k + 1][0] = in && ok0 ? (float)row[s1 + p0] : 0.f;
            pv[k + 1][1] = in && ok1 ? (float)row[s1 + p1] : 0.f;
        }
    };
    if (p.row_bf16) load_prev(reinterpret_cast<const __nv_bfloat16*>(p.prev));
    else load_prev(reinterpret_cast<const float*>(p.prev));
    float yacc[NT2][4];
#pragma unroll
    for (int j2 = 0; j2 < NT2; ++j2) {
        const float bb0 = hs == 0 ? b2_s[j2 * 8 + 2 * t] : 0.f, bb1 = hs == 0 ? b2_s[j2 * 8 + 2 * t + 1] : 0.f;
        yacc[j2][0] = bb0; yacc[j2][1] = bb1; yacc[j2][2] = bb0; yacc[j2][3] = bb1;
    }
    if constexpr (ENG == kEngTf32) {
        // mma m16n8k8.  Layer 1's accumulator fragments, after bias and activation, ARE the A fragments of layer 2 when hidden unit
        // 8j + 2t / 8j + 2t + 1 is taken as k-index t / t + 4 of k-step j (the order of the hidden units inside the sum is
        // free), so nothing moves between lanes.  bf16 weights are exact in tf32; the score row is rounded to tf32 (2^-11 relative).
        constexpr int KS1 = HQ / 8, NT1 = M_C / 8, W1_LD = M_C + 8, W2_LD = HG + 4;
        const float* w1_s = reinterpret_cast<const float*>(smem_b + lay.w1);
        const float* w2_s = reinterpret_cast<const float*>(smem_b + lay.w2);
        uint32_t afr[KS1][4];
#pragma unroll
        for (int ks = 0; ks < KS1; ++ks) {
            afr[ks][0] = to_tf32(pv[2 * ks][0]); afr[ks][1] = to_tf32(pv[2 * ks][1]);
            afr[ks][2] = to_tf32(pv[2 * ks + 1][0]); afr[ks][3] = to_tf32(pv[2 * ks + 1][1]);
        }
#pragma unroll
        for (int jj = 0; jj < (NT1 + HS - 1) / HS; ++jj) {
            const int j = jj * HS + hs;
            if (NT1 % HS != 0 && j >= NT1) break;
            float hacc[4];
            hacc[0] = hacc[2] = b1_s[j * 8 + 2 * t];
            hacc[1] = hacc[3] = b1_s[j * 8 + 2 * t + 1];
#pragma unroll
            for (int ks = 0; ks < KS1; ++ks)
                mma_tf32(hacc, afr[ks], __float_as_uint(w1_s[(ks * 8 + t) * W1_LD + j * 8 + g]), __float_as_uint(w1_s[(ks * 8 + t + 4) * W1_LD + j * 8 + g]));
            uint32_t hfr[4];
            hfr[0] = to_tf32(act_apply(hacc[0], p.act));   // (row g,   k = t)     <- column 2t
            hfr[1] = to_tf32(act_apply(hacc[2], p.act));   // (row g+8, k = t)
            hfr[2] = to_tf32(act_apply(hacc[1], p.act));   // (row g,   k = t + 4) <- column 2t + 1
            hfr[3] = to_tf32(act_apply(hacc[3], p.act));   // (row g+8, k = t + 4)
#pragma unroll
            for (int j2 = 0; j2 < NT2; ++j2)
                mma_tf32(yacc[j2], hfr, __float_as_uint(w2_s[(j * 8 + 2 * t) * W2_LD + j2 * 8 + g]), __float_as_uint(w2_s[(j * 8 + 2 * t + 1) * W2_LD + j2 * 8 + g]));
        }
    } else {
        // mma m16n8k16 on three bf16 terms of every fp32 operand: products with the bf16 weights are exact, sums are fp32
        constexpr int KP = ENG == kEngConcat ? 2 * HQ : (HQ + 15) / 16 * 16, KS1 = KP / 16;
        const __nv_bfloat16* w1_s = reinterpret_cast<const __nv_bfloat16*>(smem_b + lay.w1);
        const __nv_bfloat16* w2_s = reinterpret_cast<const __nv_bfloat16*>(smem_b + lay.w2);
        const int w1_ld = mp + 8;
        constexpr int W2_LD = HG + 8;
        uint32_t afr[KS1][3][4];
#pragma unroll
        for (int ks = 0; ks < KS1; ++ks)
#pragma unroll
            for (int q = 0; q < 4; ++q) {   // operand register q: rows g (+ 8), inputs 2t, 2t + 1 (+ 8)
                const int k8 = ks * 16 + (q & 2 ? 8 : 0), pos = q & 1 ? p1 : p0;
                float x = 0.f, y = 0.f;
                if (k8 < HQ) {
                    x = pv[k8 / 4][q & 1]; y = pv[k8 / 4 + 1][q & 1];
                } else if (ENG == kEngConcat) {
                    if (q & 1 ? ok1 : ok0) { x = s_s[(k8 - HQ + 2 * t) * CH + pos]; y = s_s[(k8 - HQ + 2 * t + 1) * CH + pos]; }
                }
                split3(x, y, afr[ks][0][q], afr[ks][1][q], afr[ks][2][q]);
            }
        const int lk = (lane & 7) + (lane & 8 ? 8 : 0), ln = lane & 16 ? 8 : 0;   // row and column half this lane addresses for ldmatrix
        for (int blk = hs; blk < mp / 16; blk += HS) {
            float hacc[2][4];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                hacc[u][0] = hacc[u][2] = b1_s[blk * 16 + u * 8 + 2 * t];
                hacc[u][1] = hacc[u][3] = b1_s[blk * 16 + u * 8 + 2 * t + 1];
            }
#pragma unroll
            for (int ks = 0; ks < KS1; ++ks) {
                uint32_t w[4];
                ldsm_x4_trans(w, w1_s + (ks * 16 + lk) * w1_ld + blk * 16 + ln);
#pragma unroll
                for (int q = 2; q >= 0; --q) {   // smallest terms first
                    mma_bf16(hacc[0], afr[ks][q], w[0], w[1]);
                    mma_bf16(hacc[1], afr[ks][q], w[2], w[3]);
                }
            }
            uint32_t hfr[3][4];
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    split3(act_apply(hacc[u][2 * e], p.act), act_apply(hacc[u][2 * e + 1], p.act), hfr[0][2 * u + e], hfr[1][2 * u + e], hfr[2][2 * u + e]);
#pragma unroll
            for (int j2 = 0; j2 < NT2; j2 += 2) {
                uint32_t w[4];
                const __nv_bfloat16* src = w2_s + (blk * 16 + lk) * W2_LD + j2 * 8;
                if (j2 + 1 < NT2) ldsm_x4_trans(w, src + ln);
                else ldsm_x2_trans(w, src);
#pragma unroll
                for (int q = 2; q >= 0; --q) {
                    mma_bf16(yacc[j2], hfr[q], w[0], w[1]);
                    if (j2 + 1 < NT2) mma_bf16(yacc[j2 + 1], hfr[q], w[2], w[3]);
                }
            }
        }
    }
    // yacc[j2]: [0] (p0, head 8 j2 + 2t), [1] (p0, + 1), [2] (p1, 2t), [3] (p1, + 1)
#pragma unroll
    for (int j2 = 0; j2 < NT2; ++j2)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int hh = j2 * 8 + 2 * t + (e & 1), pp = (e & 2) ? p1 : p0;
            if constexpr (HS == 1 && ENG != kEngConcat) s_s[hh * CH + pp] += yacc[j2][e];
            else y_s[(hs * HG + hh) * CH + pp] = yacc[j2][e];
        }
    __syncthreads();
    const size_t part = ((size_t)b * p.n_chunks + chunk) * HQ + h0;
    finish_scores<CH, HS>(p, s_s, (HS > 1 || ENG == kEngConcat) ? y_s : nullptr, ENG != kEngConcat, HG, h0, b, j0, nrows, part);
    __syncthreads();
    pv_chunk<CH>(p, s_s, reinterpret_cast<float*>(smem_b + lay.w1), b, kv0, HG, j0, nrows, p.ws_o + part * 128);
}

}  // namespace lisa
