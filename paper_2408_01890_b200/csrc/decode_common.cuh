// What the decode kernels share: their parameters and score-row access.
#pragma once
#include "common.cuh"

namespace lisa {

constexpr int kDecodeThreads = 256;
constexpr int kDecodeWarps = kDecodeThreads / 32;

struct DecodeParams {
    int B, Hq, Hkv, d, L_cap, L_uniform, n_chunks;
    int chunk;              // cached positions per chunk: 128, or 64 or 32 in the kernels for small batches
    int heads;              // query heads per CTA where the heads are divided over CTAs
    int prefetch;           // a CTA asks its K or K' and V of this many of its KV heads into L2 when it starts; -1: nothing
    int late_release;       // the merge lets its successor in behind its wait, not at its start (see merge_releases_late)
    int least, most;        // dealt chunks (see decode_item): the launch does its work only if least..most of them hold positions (see launch_shared_fast)
    const int32_t* seq_lens;
    // shared layer
    const void* prev;       // fp32, or bf16 when row_bf16
    int64_t prev_sb, prev_sh;
    TView qp;
    const void* kpT;
    int r, m, act, integrate, ffn_layers, w_dtype;
    const void *w1, *b1, *w2, *b2;
    int w_vec;              // W1 and W2 are bf16 and 16-byte aligned
    // standard layer
    TView q;
    const void* kcache;
    // common
    const void* vcache;
    int cache_dtype;
    void* out_scores;       // fp32, or bf16 when row_bf16
    int64_t sc_sb, sc_sh;
    int row_bf16;           // the score rows handed between layers are bf16 (Sec. 5.2 counts them at 2 bytes) instead of fp32
    float *ws_m, *ws_l, *ws_o;
    TView o;
};

// Score-row access: RB = rows are bf16.
template <bool RB>
__device__ __forceinline__ float ld_row(const void* p, int64_t i) {
    if constexpr (RB) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[i]);
    else return reinterpret_cast<const float*>(p)[i];
}
template <bool RB>
__device__ __forceinline__ void st_row(void* p, int64_t i, float v) {
    if constexpr (RB) reinterpret_cast<__nv_bfloat16*>(p)[i] = __float2bfloat16_rn(v);
    else reinterpret_cast<float*>(p)[i] = v;
}

__device__ __forceinline__ float ldw(const void* p, int idx, int dtype) { return p ? ld_elem(p, idx, dtype) : 0.f; }

__device__ __forceinline__ uint4 ld_stream16(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// The same where `ok`, else zeros: one predicated load, no branch
__device__ __forceinline__ uint4 ld_stream16_or_zero(const void* p, bool ok) {
    uint4 v;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
                 "mov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\tmov.b32 %3, 0;\n\t"
                 "@q ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n\t}"
                 : "=&r"(v.x), "=&r"(v.y), "=&r"(v.z), "=&r"(v.w)
                 : "l"(p), "r"((int)ok));
    return v;
}

__device__ __forceinline__ void bf16x8_to_f32(const uint4& v, float* f) {
    f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xffff0000u);
    f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xffff0000u);
    f[4] = __uint_as_float(v.z << 16); f[5] = __uint_as_float(v.z & 0xffff0000u);
    f[6] = __uint_as_float(v.w << 16); f[7] = __uint_as_float(v.w & 0xffff0000u);
}

// Context length of sequence b, never beyond the chunks the launch covers.
__device__ __forceinline__ int decode_length(const DecodeParams& p, int b) {
    return p.seq_lens ? min(p.seq_lens[b], p.L_uniform) : p.L_uniform;
}

// A CTA's sequence, chunk and context length; false if there is none for it.  Uniform batches: the grid's coordinates.  Ragged ones: the
// chunks that hold positions, numbered over all sequences, go to the first CTAs of the grid, which the hardware spreads evenly; with
// the grid's coordinates those without a chunk leave at once and the others pile up (16 sequences of up to 2900 positions: 210 CTAs with
// work on 112 of 148 SMs, three on 27 of them).  Every warp counts for itself, 32 sequences at a time, all lengths in flight together.
constexpr int kDenseMaxB = 128;
template <int CH, bool DENSE>
__device__ __forceinline__ bool decode_item(const DecodeParams& p, int& b, int& chunk, int& L) {
    b = blockIdx.z;
    chunk = blockIdx.x;
    if constexpr (!DENSE) {
        L = decode_length(p, b);
        return chunk * CH < L;
    }
    const int lane = threadIdx.x & 31, at = blockIdx.z * gridDim.x + blockIdx.x;
    int len[kDenseMaxB / 32];
#pragma unroll
    for (int q = 0; q < kDenseMaxB / 32; ++q) {
        const int s = q * 32 + lane;
        len[q] = s < p.B ? max(0, min(p.seq_lens[s], p.L_uniform)) : 0;
    }
    int count = 0;                                                    // chunks of the sequences before 32 q, in the end of all
    bool found = false;
#pragma unroll
    for (int q = 0; q < kDenseMaxB / 32; ++q) {
        if (q * 32 >= p.B) break;
        const int n = (len[q] + CH - 1) / CH, left = at - count;
        int upto = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += v;
        }
        const uint32_t above = __ballot_sync(0xffffffffu, upto > left);
        if (above && !found) {
            const int src = __ffs(above) - 1;
            b = __shfl_sync(0xffffffffu, q * 32 + src, 0);   // (uniform, as the compiler sees it)
            chunk = __shfl_sync(0xffffffffu, left - (upto - n), src);
            L = __shfl_sync(0xffffffffu, len[q], src);
            found = true;
        }
        count += __shfl_sync(0xffffffffu, upto, 31);
    }
    return found && count >= p.least && count <= p.most;
}

}  // namespace lisa
