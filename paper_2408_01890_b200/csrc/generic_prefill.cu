// General SIMT prefill of a LiSA shared layer (and, with chain_len == 0, of a standard layer).
//
// One CTA per query row (b, i).  Keys are visited in chunks of 128, whose score chain is rebuilt in fp32: the anchor score
// q0.k0/sqrt(d) for every head (Eq. 2), then per link the low-rank difference q'.k'/sqrt(r) (Eq. 3), the head-axis FFN and the
// integration (Sec. 5.1, Eq. 4).  The chunk's final scores get the causal mask (keys j > i are never visited), an online softmax
// per head, and the product with V (Eq. 1).  The N x N x Hq scores are never stored.  Every integrate mode, activation, FFN depth,
// dtype and shape in the supported range runs here; the tensor-core kernels cover the fast cases.
//
// A small prompt is bound by the latency of one CTA, so every phase spreads over all threads with its loads in flight together: the dot
// products over (head, key, part of the row), the FFN over keys and hidden units (weights in shared memory; 2, 4 or 8 heads in registers), the softmax over heads, the
// product with V over (head, column) and, where these are few, ranges of keys.  How far that goes without costing resident CTAs depends on the
// grid and the type, see kOverHeads below.  4 heads of 32, N 128, fp32, the standard layer and a shared one back to back 17.6 us (22.7 as kOverHeads).
#include "common.cuh"

namespace lisa {
namespace {

constexpr int kChunk = 128;
constexpr int kMaxThreads = 512;   // a grid that leaves SMs idle runs with twice the threads of a larger one

struct PrefillParams {
    int B, N, Hq, Hkv, d, c;
    TView q0, k0, v, o;
    LinkDev links[kMaxChain];
    int vec_k0, vec_kp[kMaxChain];   // rows start on 16 bytes (fp32 and bf16 builds)
    int w_off[kMaxChain], w_floats[kMaxChain];   // where a link's weights are staged in shared memory (floats; -1: read from memory), how many
};

// A CTA's shared memory, in floats from its start; the staged weights follow.  q0, and q' of every link, are read as float4 (dots<0, 4>) at
// h * d and h * kMaxRank, so both must start on 16 bytes whatever the head count: they come before the arrays of Hq values.
struct SmemLayout {
    int q0, o, s, d, qp, m, l, sc, total;
    __host__ __device__ constexpr SmemLayout(int Hq, int width, int c)
        : q0(0),                          // [Hq][d]
          o(q0 + Hq * width),             // [Hq][d]
          s(o + Hq * width),              // [Hq][kChunk] scores of the chunk
          d(s + Hq * kChunk),             // [Hq][kChunk] a link's difference; then partial sums of the product with V
          qp(d + Hq * kChunk),            // [c][Hq][kMaxRank]
          m(qp + c * Hq * kMaxRank),      // [Hq]
          l(m + Hq),                      // [Hq]
          sc(l + Hq),                     // [Hq]
          total(sc + Hq) {}
};
constexpr bool vectors_aligned() {
    for (int Hq = 1; Hq <= kMaxHeads; ++Hq)
        for (int width = 32; width <= 128; width *= 2)
            for (int c = 0; c <= kMaxChain; ++c)
                if (SmemLayout(Hq, width, c).q0 % 4 != 0 || SmemLayout(Hq, width, c).qp % 4 != 0) return false;
    return kMaxRank % 4 == 0;
}
static_assert(vectors_aligned(), "float4 reads of q0 and q' need 16-byte aligned rows");

// DT: 0 = fp32, 1 = bf16, 2 = any mix, decided per access
template <int DT>
__device__ __forceinline__ float ld(const TView& t, int64_t i) {
    if constexpr (DT == 0) return reinterpret_cast<const float*>(t.ptr)[i];
    else if constexpr (DT == 1) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(t.ptr)[i]);
    else return ld_elem(t.ptr, i, t.dtype);
}

// How a CTA's phases are laid out.
//   kOverHeads  rows of K numbered head by head, four of a lane in flight; a thread to a position's FFN.  Every bf16 or mixed call, and head counts
//               known at run time.
//   kWide       rows numbered key by key, eight of a lane in flight; hidden units over the lanes a position has to spare; V ahead of the product.
//               Twice the registers: one CTA of 512 threads to an SM, two of 256.
//   kResident   as kWide with four rows of a lane and V behind the softmax: 64 registers, twice the CTAs.
// fp32 takes kWide where one CTA per SM is all there is, and for one prompt of up to three rows per SM, whose later CTAs are the short rows;
// elsewhere kResident.  One link, heads of 32, us, kOverHeads | kWide | kResident:
//   fp32, 4 heads   128 rows 12.1 | 10.2 | -     400 44.8 | 37.9 | 46.5    2 x 80 12.0 | 16.9 | 11.8    2 x 1000 223 | 310 | 230
//   fp32, 8 heads   128 rows 16.0 | 16.2 | -     400 67.7 | 67.2 | 86.6    2 x 80 22.3 | 20.3 | 16.7    2 x 1000 525 | 535 | 435
//   bf16, 4 heads   128 rows 11.1 | 12.7 | -     400 38.9 | 38.3 | 47.0    2 x 80 11.0 | 18.1 | 11.6    2 x 1000 189 | 293 | 224
//   bf16, 8 heads   128 rows 14.9 | 18.6 | -     400 57.4 | 79.0 | 117     2 x 80 19.8 | 21.7 | 19.3    2 x 1000 445 | 638 | 573
// (Prompts between lose up to 14 % to kOverHeads at 4 heads of 32, 148 rows 15.0 | 16.9 and 296 rows 28.8 | 32.9 | 30.4, and gain as much at heads of
// 64, 200 rows 28.8 | 22.1 | 27.4; 2 heads 400 rows 24.0 | 26.8 | 28.3, 2 x 1000 180 | 211 | 135.)
constexpr int kOverHeads = 0, kWide = 1, kResident = 2;

// out[h][jj] = scale * (q[h] . row of key jj in KV head h / G) for the chunk's nk keys: neighbouring lanes take neighbouring V values of a
// row (V values are 16 bytes, or one where rows do not start on 16 bytes), several rows of a lane are in flight, shuffles add up a row.  Numbered
// key by key, a chunk of few keys takes few rounds; head by head spares the divisions where the head count is known at run time (6 heads of
// 64, 300 positions 115 us, 162 the other way).
template <int DT, int V, int HQ, int FORM>
__device__ __forceinline__ void dots(float* out, const float* q, int q_ld, const TView& t, int64_t at, int Hq, int G, int nk, int n, float scale) {
    constexpr bool KEYS = FORM != kOverHeads;
    constexpr int U = FORM == kWide ? 8 : 4;
    const int lanes = (n + V - 1) / V;
    const int lpr = lanes <= 1 ? 1 : lanes >= 32 ? 32 : 1 << (32 - __clz(lanes - 1));   // lanes per row
    const int sub = threadIdx.x & (lpr - 1), grp = threadIdx.x / lpr, groups = blockDim.x / lpr, total = Hq * (KEYS ? nk : kChunk);
    for (int r0 = 0; r0 < total; r0 += U * groups) {
        float part[U];
        int64_t row[U];
        const float* qh[U];
        bool ok[U];
        int o[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int rr = r0 + u * groups + grp, jj = KEYS ? rr / Hq : rr % kChunk, h = KEYS ? rr - jj * Hq : rr / kChunk;
            ok[u] = rr < total && jj < nk;
            row[u] = at + jj * t.sn + (G == 1 ? h : h / G) * t.sh;
            qh[u] = q + h * q_ld;
            o[u] = h * kChunk + jj;
            part[u] = 0.f;
        }
        for (int x = sub * V; x < n; x += lpr * V) {   // (once, unless rows of more than 32 values are read one by one)
            if constexpr (V == 4) {
                float4 v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = ok[u] ? *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(t.ptr) + row[u] + x) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (!ok[u]) continue;
                    const float4 w = *reinterpret_cast<const float4*>(qh[u] + x);
                    part[u] = fmaf(w.x, v[u].x, part[u]); part[u] = fmaf(w.y, v[u].y, part[u]);
                    part[u] = fmaf(w.z, v[u].z, part[u]); part[u] = fmaf(w.w, v[u].w, part[u]);
                }
            } else if constexpr (V == 8) {
                uint4 v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = ok[u] ? *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(t.ptr) + row[u] + x) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (!ok[u]) continue;
                    const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        part[u] = fmaf(qh[u][x + 2 * j], __uint_as_float(w[j] << 16), part[u]);
                        part[u] = fmaf(qh[u][x + 2 * j + 1], __uint_as_float(w[j] & 0xffff0000u), part[u]);
                    }
                }
            } else {
                float v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = ok[u] ? ld<DT>(t, row[u] + x) : 0.f;
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (ok[u]) part[u] = fmaf(qh[u][x], v[u], part[u]);
            }
        }
        for (int off = lpr >> 1; off > 0; off >>= 1)
#pragma unroll
            for (int u = 0; u < U; ++u) part[u] += __shfl_xor_sync(0xffffffffu, part[u], off);
        if (sub == 0)
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (ok[u]) out[o[u]] = part[u] * scale;
    }
}
template <int DT, int HQ, int FORM>
__device__ __forceinline__ void dots_any(float* out, const float* q, int q_ld, const TView& t, int64_t at, int Hq, int G, int nk, int n, float scale, int vec) {
    if (DT == 0 && vec && n % 4 == 0) dots<DT, DT == 0 ? 4 : 1, HQ, FORM>(out, q, q_ld, t, at, Hq, G, nk, n, scale);
    else if (DT == 1 && vec && n % 8 == 0) dots<DT, DT == 1 ? 8 : 1, HQ, FORM>(out, q, q_ld, t, at, Hq, G, nk, n, scale);
    else dots<DT, 1, HQ, FORM>(out, q, q_ld, t, at, Hq, G, nk, n, scale);
}

// A link's FFN weights: fp32 in shared memory (SM; w1, b1, w2, b2 one after the other), or where the model keeps them.
template <bool SM>
struct Weights {
    const float *p1, *pb1, *p2, *pb2;
    const LinkDev& l;
    __device__ Weights(const float* s, const LinkDev& link, int h_in, int Hq) : p1(s), pb1(s + h_in * link.m), p2(pb1 + link.m), pb2(p2 + link.m * Hq), l(link) {}
    __device__ __forceinline__ float w1(int i) const { return SM ? p1[i] : ld_elem(l.w1, i, l.w_dtype); }
    __device__ __forceinline__ float b1(int i) const { return SM ? pb1[i] : l.b1 ? ld_elem(l.b1, i, l.w_dtype) : 0.f; }
    __device__ __forceinline__ float w2(int i) const { return SM ? p2[i] : ld_elem(l.w2, i, l.w_dtype); }
    __device__ __forceinline__ float b2(int i) const { return SM ? pb2[i] : l.b2 ? ld_elem(l.b2, i, l.w_dtype) : 0.f; }
};

// Sec. 5.1 at one position: a <- Integrate(Align(a), dl); a and dl are columns of shared memory, one head every kChunk floats.  HQ > 0: that
// many heads, in registers, and the hidden units over `parts` neighbouring lanes (all lanes of the warp come here; lanes without a
// position of their own write nothing).
template <int HQ, bool SM>
__device__ __forceinline__ void align_integrate(float* a, const float* dl, int n_heads, const Weights<SM>& w, int part, int parts, bool write) {
    const int Hq = HQ ? HQ : n_heads;
    const LinkDev& lk = w.l;
    if (lk.integrate == LISA_INTEGRATE_PLUS) {
        if (write)
            for (int g = 0; g < Hq; ++g) a[g * kChunk] += dl[g * kChunk];
        return;
    }
    const int m = lk.m;
    const bool concat = lk.integrate == LISA_INTEGRATE_CONCAT, two = lk.ffn_layers == 2;
    const int act = lk.act;
    constexpr int CAP = HQ ? HQ : kMaxHeads;
    float x[CAP], y[CAP];
#pragma unroll(HQ ? HQ : 1)
    for (int h = 0; h < Hq; ++h) {
        x[h] = a[h * kChunk];
        y[h] = two && part == 0 ? w.b2(h) : 0.f;
    }
    auto units = [&](auto activate) {
#pragma unroll(HQ ? 4 : 1)
        for (int u = part; u < m; u += parts) {
            float s = w.b1(u);
#pragma unroll(HQ ? HQ : 4)
            for (int h = 0; h < Hq; ++h) s = fmaf(x[h], w.w1(h * m + u), s);
            if (concat)
#pragma unroll(HQ ? HQ : 4)
                for (int h = 0; h < Hq; ++h) s = fmaf(dl[h * kChunk], w.w1((Hq + h) * m + u), s);
            if (two) {
                s = activate(s);
#pragma unroll(HQ ? HQ : 4)
                for (int g = 0; g < Hq; ++g) y[g] = fmaf(s, w.w2(u * Hq + g), y[g]);
            } else if constexpr (HQ > 0) {
#pragma unroll
                for (int g = 0; g < HQ; ++g) y[g] = g == u ? s : y[g];
            } else {
                y[u] = s;   // one layer: m == Hq
            }
        }
    };
    const float floor = act == LISA_ACT_RELU ? 0.f : -INFINITY;
    if (act == LISA_ACT_SILU) units([](float s) { return act_apply(s, LISA_ACT_SILU); });
    else units([floor](float s) { return fmaxf(s, floor); });
    if constexpr (HQ > 0) {
        for (int off = parts >> 1; off > 0; off >>= 1)
#pragma unroll
            for (int g = 0; g < HQ; ++g) y[g] += __shfl_xor_sync(0xffffffffu, y[g], off);
    }
    if (!write) return;
#pragma unroll(HQ ? HQ : 1)
    for (int g = 0; g < Hq; ++g) a[g * kChunk] = lk.integrate == LISA_INTEGRATE_ADD ? y[g] + dl[g * kChunk] : y[g];
}

template <int DT, int HQ, int FORM>
__global__ void __launch_bounds__(kMaxThreads, FORM == kResident ? 2 : 0) generic_prefill_kernel(const __grid_constant__ PrefillParams p) {
    extern __shared__ __align__(16) float smem[];
    const int b = blockIdx.y, i = (int)(gridDim.x - 1 - blockIdx.x), tid = threadIdx.x;   // the longest rows first
    const int Hq = HQ ? HQ : p.Hq, d = p.d, G = Hq / p.Hkv;
    const int warp = tid >> 5, lane = tid & 31, kThreads = blockDim.x, kWarps = kThreads / 32;
    const SmemLayout at(Hq, d, p.c);
    float *q0_s = smem + at.q0, *o_s = smem + at.o, *s_s = smem + at.s, *d_s = smem + at.d, *qp_s = smem + at.qp;
    float *m_s = smem + at.m, *l_s = smem + at.l, *sc_s = smem + at.sc;

    // everything a CTA reads once, as one flat range: one round of loads for a small layer, not one per tensor
    chain_release();
    chain_wait();
    const int n_q0 = Hq * d;
    int total = n_q0;
    for (int k = 0; k < p.c; ++k) total += Hq * p.links[k].r + p.w_floats[k];
    for (int e0 = tid; e0 < total; e0 += kThreads) {
        int e = e0;
        if (e < n_q0) {
            const int h = e / d, x = e % d;
            q0_s[e] = ld<DT>(p.q0, b * p.q0.sb + i * p.q0.sn + h * p.q0.sh + x);
            o_s[e] = 0.f;
            continue;
        }
        e -= n_q0;
        int k = 0;
        while (e >= Hq * p.links[k].r + p.w_floats[k]) e -= Hq * p.links[k].r + p.w_floats[k++];
        const LinkDev& lk = p.links[k];
        if (e < Hq * lk.r) {
            const int h = e / lk.r, x = e % lk.r;
            qp_s[k * Hq * kMaxRank + h * kMaxRank + x] = ld<DT>(lk.qp, b * lk.qp.sb + i * lk.qp.sn + h * lk.qp.sh + x);
            continue;
        }
        e -= Hq * lk.r;   // w1, b1, w2, b2 one after the other
        const int n1 = (lk.integrate == LISA_INTEGRATE_CONCAT ? 2 : 1) * Hq * lk.m, n2 = lk.m * Hq;
        float v;
        if (e < n1) v = ld_elem(lk.w1, e, lk.w_dtype);
        else if (e < n1 + lk.m) v = lk.b1 ? ld_elem(lk.b1, e - n1, lk.w_dtype) : 0.f;
        else if (e < n1 + lk.m + n2) v = ld_elem(lk.w2, e - n1 - lk.m, lk.w_dtype);
        else v = lk.b2 ? ld_elem(lk.b2, e - n1 - lk.m - n2, lk.w_dtype) : 0.f;
        smem[p.w_off[k] + e] = v;
    }
    for (int h = tid; h < Hq; h += kThreads) {
        m_s[h] = -INFINITY;
        l_s[h] = 0.f;
    }
    __syncthreads();

    const float inv_sqrt_d = rsqrtf((float)d);
    // the product with V: a thread owns output columns, or, where there are fewer of these than threads, one column and a range of keys
    const int cols = Hq * d, splits = cols < kThreads ? min(kThreads / cols, max(1, Hq * kChunk / cols)) : 1;
    for (int j0 = 0; j0 <= i; j0 += kChunk) {
        const int nk = min(kChunk, i + 1 - j0);
        dots_any<DT, HQ, FORM>(s_s, q0_s, d, p.k0, b * p.k0.sb + (int64_t)j0 * p.k0.sn, Hq, G, nk, d, inv_sqrt_d, p.vec_k0);
        // where a thread has one column and a short range of keys, its values of V come now, under the phases before the product
        constexpr int VA = 32;
        const int v_part = tid / cols, v_col = tid - v_part * cols, v0 = nk * v_part / splits, v1 = nk * (v_part + 1) / splits;
        const bool ahead = FORM == kWide && splits > 1 && (nk + splits - 1) / splits <= VA;
        float va[VA];
        if (ahead && v_part < splits) {
            const int h = v_col / d;
            const int64_t vb = b * p.v.sb + (int64_t)(j0 + v0) * p.v.sn + (h / G) * p.v.sh + (v_col - h * d);
#pragma unroll
            for (int q = 0; q < VA; ++q) va[q] = v0 + q < v1 ? ld<DT>(p.v, vb + (int64_t)q * p.v.sn) : 0.f;
        }
        for (int k = 0; k < p.c; ++k) {
            const LinkDev& lk = p.links[k];
            dots_any<DT, HQ, FORM>(d_s, qp_s + k * Hq * kMaxRank, kMaxRank, lk.kp, b * lk.kp.sb + (int64_t)j0 * lk.kp.sn, Hq, G, nk, lk.r, rsqrtf((float)lk.r), p.vec_kp[k]);
            __syncthreads();
            const int h_in = (lk.integrate == LISA_INTEGRATE_CONCAT ? 2 : 1) * Hq;
            if (FORM != kOverHeads || tid < nk) {
                const int parts = FORM != kOverHeads ? kThreads / kChunk : 1, pos = tid / parts, part = tid - pos * parts;
                const bool write = part == 0 && pos < nk;
                if (p.w_off[k] >= 0) align_integrate<HQ>(s_s + pos, d_s + pos, Hq, Weights<true>(smem + p.w_off[k], lk, h_in, Hq), part, parts, write);
                else align_integrate<HQ>(s_s + pos, d_s + pos, Hq, Weights<false>(nullptr, lk, h_in, Hq), part, parts, write);
            }
            __syncthreads();
        }
        if (p.c == 0) __syncthreads();
        for (int h = warp; h < Hq; h += kWarps) {
            float v[kChunk / 32];
            float cmax = -INFINITY;
#pragma unroll
            for (int t = 0; t < kChunk / 32; ++t) {
                v[t] = lane + 32 * t < nk ? s_s[h * kChunk + lane + 32 * t] : -INFINITY;   // causal mask, after the chain
                cmax = fmaxf(cmax, v[t]);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, off));
            const float m_old = m_s[h];
            const float m_new = fmaxf(m_old, cmax);
            float sum = 0.f;
#pragma unroll
            for (int t = 0; t < kChunk / 32; ++t) {
                const float e = __expf(v[t] - m_new);
                s_s[h * kChunk + lane + 32 * t] = e;
                sum += e;
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
            __syncwarp();
            if (lane == 0) {
                const float sc = __expf(m_old - m_new);
                sc_s[h] = sc;
                l_s[h] = l_s[h] * sc + sum;
                m_s[h] = m_new;
            }
        }
        __syncthreads();
        if (ahead) {
            if (v_part < splits) {
                const float* e_s = s_s + v_col / d * kChunk + v0;
                float acc = 0.f;
#pragma unroll
                for (int q = 0; q < VA; ++q)
                    if (v0 + q < v1) acc = fmaf(e_s[q], va[q], acc);
                d_s[tid] = acc;
            }
        } else for (int e = tid; e < cols * splits; e += kThreads) {
            const int part = e / cols, col = e % cols, h = col / d, x = col % d;
            const int k0 = nk * part / splits, k1 = nk * (part + 1) / splits;
            const int64_t vb = b * p.v.sb + (int64_t)j0 * p.v.sn + (h / G) * p.v.sh + x;
            float acc = 0.f;
#pragma unroll 16
            for (int jj = k0; jj < k1; ++jj) acc = fmaf(s_s[h * kChunk + jj], ld<DT>(p.v, vb + (int64_t)jj * p.v.sn), acc);
            if (splits == 1) o_s[col] = o_s[col] * sc_s[h] + acc;
            else d_s[e] = acc;
        }
        __syncthreads();
        if (splits > 1) {
            if (tid < cols) {
                float acc = o_s[tid] * sc_s[tid / d];
                for (int q = 0; q < splits; ++q) acc += d_s[q * cols + tid];
                o_s[tid] = acc;
            }
            __syncthreads();
        }
    }
    for (int e = tid; e < cols; e += kThreads) {
        const int h = e / d, x = e % d;
        st_elem(const_cast<void*>(p.o.ptr), b * p.o.sb + i * p.o.sn + h * p.o.sh + x, p.o.dtype, o_s[e] / l_s[h]);
    }
}

constexpr size_t kMaxSmemFloats = 232448 / sizeof(float);

bool vec_rows(const lisa_tensor& t) {
    const int64_t n = t.dtype == LISA_BF16 ? 8 : 4;
    return t.stride_b % n == 0 && t.stride_n % n == 0 && t.stride_h % n == 0;   // (the pointer is: checked by the entry points)
}

// Head counts a compile-time constant keeps a position's scores in registers for; every other count runs the loops over local memory.
// One link, heads of 32, fp32, 128 positions: 2 heads 8.9 us (loops 10.3), 4 heads 11.9 (13.0), 8 heads 15.9 (21.9); two
// sequences of 1000, 8 heads: 525 (720).  Counts of tiny test and draft models; beyond eight, larger models are the tensor-core kernels'.
template <int DT, int FORM>
void* pick(int Hq) {
    return Hq == 2   ? reinterpret_cast<void*>(generic_prefill_kernel<DT, 2, FORM>)
           : Hq == 4 ? reinterpret_cast<void*>(generic_prefill_kernel<DT, 4, FORM>)
           : Hq == 8 ? reinterpret_cast<void*>(generic_prefill_kernel<DT, 8, FORM>)
                     : reinterpret_cast<void*>(generic_prefill_kernel<DT, 0, kOverHeads>);
}

}  // namespace

cudaError_t launch_generic_prefill(const lisa_shared_prefill_args& a, cudaStream_t s) {
    PrefillParams p;
    p.B = a.B; p.N = a.N; p.Hq = a.Hq; p.Hkv = a.Hkv; p.d = a.d; p.c = a.chain_len;
    p.q0 = make_view(a.q0); p.k0 = make_view(a.k0); p.v = make_view(a.v); p.o = make_view(a.o);
    p.vec_k0 = vec_rows(a.k0);
    int dt = a.q0.dtype;
    bool same = a.k0.dtype == dt && a.v.dtype == dt;
    size_t floats = SmemLayout(a.Hq, a.d, a.chain_len).total;
    for (int k = 0; k < a.chain_len; ++k) {
        const lisa_link& l = a.links[k];
        p.links[k] = make_link(l);
        p.vec_kp[k] = vec_rows(l.kp);
        same = same && l.qp.dtype == dt && l.kp.dtype == dt;
        p.w_off[k] = -1;
        p.w_floats[k] = 0;
        if (l.integrate == LISA_INTEGRATE_PLUS) continue;
        // staged while a CTA keeps to half an SM's shared memory (or is beyond that anyway)
        const size_t n = (size_t)(l.integrate == LISA_INTEGRATE_CONCAT ? 2 : 1) * a.Hq * l.m + l.m + (l.ffn_layers == 2 ? (size_t)l.m * a.Hq + a.Hq : 0);
        const size_t room = floats > kMaxSmemFloats / 2 - 512 ? kMaxSmemFloats : kMaxSmemFloats / 2 - 512;
        if (floats + n <= room) { p.w_off[k] = (int)floats; p.w_floats[k] = (int)n; floats += n; }
    }
    const int64_t rows = (int64_t)a.N * a.B, sms = sm_count();
    const bool wide = rows <= sms || (a.B == 1 && rows <= 3 * sms);
    const void* kernel = !same ? pick<2, kOverHeads>(a.Hq) : dt == LISA_BF16 ? pick<1, kOverHeads>(a.Hq) : wide ? pick<0, kWide>(a.Hq) : pick<0, kResident>(a.Hq);
    const size_t smem = floats * sizeof(float);
    cudaError_t e = allow_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    const int threads = rows <= 2 * sms ? kMaxThreads : kMaxThreads / 2;
    e = launch_chained(reinterpret_cast<void (*)(PrefillParams)>(const_cast<void*>(kernel)), dim3(a.N, a.B), dim3(threads), smem, s, p);
    count_launches(1);
    return e;
}

}  // namespace lisa
