// Cache append (Sec. 2.2 "KV cache"; Sec. 5.2: a shared layer stores K_LR in place of K).
// STANDARD layers keep K as [B][Hkv][L_cap][d]; SHARED layers keep K' transposed, [B][Hkv][r][L_cap],
// so that the decode kernel reads full 16-byte vectors along the position axis whatever r is.
#include <algorithm>

#include "common.cuh"

namespace lisa {
namespace {

struct AppendParams {
    int B, Hkv, L_cap, d, r, n_new, kind, dtype;
    TView k, v;
    void* kc;
    void* vc;
    const int32_t* lens_before;
    int* status;
};

// rows of d elements (V, or K of a STANDARD layer): 16 bytes per lane, four vectors of a thread in flight.  Bound by HBM once the
// vectors are: 2 x 1777 positions of 40 heads (K and V) 26 us, 33 with one in flight and 64-bit index divisions.
template <typename Vec, int kElems>
__device__ __forceinline__ void append_rows(const AppendParams& p, const TView& src, void* dst_base, bool count_drops) {
    constexpr int U = 4;
    const uint32_t vec_per_row = p.d / kElems;      // a power of two: 4 ... 32
    const int shift = 31 - __clz(vec_per_row);
    const int64_t total = (int64_t)p.B * p.n_new * p.Hkv * vec_per_row, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e0 < total; e0 += U * step) {
        Vec val[U];
        Vec* dp[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t e = e0 + u * step;
            dp[u] = nullptr;
            if (e >= total) continue;
            const uint32_t vi = (uint32_t)e & (vec_per_row - 1), row = (uint32_t)(e >> shift);   // rows < 2^31: checked by the launch
            const uint32_t tb = row / (uint32_t)p.Hkv, g = row - tb * p.Hkv, b = tb / (uint32_t)p.n_new, t = tb - b * p.n_new;
            const int64_t pos = (int64_t)(p.lens_before ? p.lens_before[b] : 0) + t;
            if (pos >= p.L_cap || pos < 0) {
                if (count_drops && vi == 0 && g == 0) atomicAdd(p.status, 1);
                continue;
            }
            const char* sp = reinterpret_cast<const char*>(src.ptr) +
                             (b * src.sb + t * src.sn + g * src.sh) * (int64_t)(sizeof(Vec) / kElems) + (int64_t)vi * sizeof(Vec);
            val[u] = *reinterpret_cast<const Vec*>(sp);
            dp[u] = reinterpret_cast<Vec*>(dst_base) + (((int64_t)b * p.Hkv + g) * p.L_cap + pos) * vec_per_row + vi;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (dp[u]) *dp[u] = val[u];
    }
}

// K' of a SHARED layer, few new positions: one thread per value, so that no load waits for another (a thread that copied a head's r
// values one after the other took 8 us for a decode step)
template <typename T>
__device__ __forceinline__ void append_kp_transposed(const AppendParams& p) {
    const int64_t total = (int64_t)p.B * p.n_new * p.Hkv * p.r;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t row = total >> 31 ? (uint32_t)(e / p.r) : (uint32_t)e / (uint32_t)p.r;   // 64-bit division only where it must be
        const uint32_t x = (uint32_t)(e - (int64_t)row * p.r), tb = row / (uint32_t)p.Hkv, g = row - tb * p.Hkv;
        const uint32_t b = tb / (uint32_t)p.n_new, t = tb - b * p.n_new;
        const int64_t pos = (int64_t)(p.lens_before ? p.lens_before[b] : 0) + t;
        if (pos >= p.L_cap || pos < 0) continue;  // counted by the V rows
        reinterpret_cast<T*>(p.kc)[(((int64_t)b * p.Hkv + g) * p.r + x) * p.L_cap + pos] =
            reinterpret_cast<const T*>(p.k.ptr)[b * p.k.sb + t * p.k.sn + g * p.k.sh + x];
    }
}

// The same for a prompt: 64 positions x HB heads at a time through shared memory, so that the rows of r values are read as they lie
// (neighbouring threads reading them r values apart cost 32 requests per load) and written along the positions.  Bound by the latency
// of its loads, so a warp has all of its eight positions' in flight.
constexpr int kTilePos = 64, kAppendThreads = 256;
template <typename T>
__device__ __forceinline__ void append_kp_tiled(const AppendParams& p) {
    constexpr int HB = 2, LD = kTilePos + (sizeof(T) == 2 ? 2 : 1), NW = kAppendThreads / 32, K = HB * kMaxRank / 32, U = kTilePos / NW;
    __shared__ T tile[HB * kMaxRank * LD];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tn = (p.n_new + kTilePos - 1) / kTilePos, tg = (p.Hkv + HB - 1) / HB, r = p.r;
    for (int tl = blockIdx.x; tl < p.B * tn * tg; tl += gridDim.x) {
        const int g0 = tl % tg * HB, t0 = tl / tg % tn * kTilePos, b = tl / tg / tn;
        const int heads = min(HB, p.Hkv - g0), cnt = min(kTilePos, p.n_new - t0), vals = heads * r;
        const int64_t pos0 = (int64_t)(p.lens_before ? p.lens_before[b] : 0) + t0;
        const T* src = reinterpret_cast<const T*>(p.k.ptr) + b * p.k.sb + (t0 + warp) * p.k.sn + g0 * p.k.sh;
        T v[K][U];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int e = lane + 32 * k, g = e / r;
            const T* sp = src + g * p.k.sh + (e - g * r);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (e < vals && warp + u * NW < cnt) v[k][u] = sp[u * NW * p.k.sn];
        }
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (lane + 32 * k < vals) tile[(lane + 32 * k) * LD + warp + u * NW] = v[k][u];
        __syncthreads();
        T* dst = reinterpret_cast<T*>(p.kc) + ((int64_t)b * p.Hkv + g0) * r * p.L_cap + pos0;   // (head, rank row) = g0 * r + e
#pragma unroll 4
        for (int e = warp; e < vals; e += NW)
#pragma unroll
            for (int t = lane; t < kTilePos; t += 32)
                if (t < cnt && pos0 + t >= 0 && pos0 + t < p.L_cap) dst[(int64_t)e * p.L_cap + t] = tile[e * LD + t];
        __syncthreads();
    }
}

// One launch appends both halves of a layer's cache: blockIdx.y = 1 the V rows, 0 the K rows (STANDARD) or the transposed K_LR
// columns (SHARED), whose CTAs wait longer and therefore go first.  Four CTAs per SM: the tiled copy's registers must not cost the
// V rows their loads in flight (at two per SM 2 x 1777 positions of 40 heads took 36 instead of 26 us).
template <typename Vec, int kElems, typename T>
__global__ void __launch_bounds__(kAppendThreads, 4) append_kernel(const __grid_constant__ AppendParams p) {
    chain_release();
    chain_wait();
    if (blockIdx.y == 1) append_rows<Vec, kElems>(p, p.v, p.vc, true);
    else if (p.kind == LISA_CACHE_STANDARD) append_rows<Vec, kElems>(p, p.k, p.kc, false);
    else if (p.n_new >= kTilePos) append_kp_tiled<T>(p);
    else append_kp_transposed<T>(p);
}

}  // namespace

cudaError_t launch_kvcache_append(const lisa_kvcache_layer& c, const lisa_tensor& k, const lisa_tensor& v,
                                  const int32_t* lens_before, int n_new, cudaStream_t s) {
    AppendParams p{c.B, c.Hkv, c.L_cap, c.d, c.r, n_new, c.kind, c.dtype, make_view(k), make_view(v), c.k, c.v,
                   lens_before, status_words()};
    if (!p.status) return cudaErrorUnknown;
    const int threads = kAppendThreads;
    const int64_t rows = (int64_t)c.B * n_new * c.Hkv;
    if (rows > 0x7fffffff) return cudaErrorInvalidValue;   // (137 GB of V at the narrowest width, and as much again in the cache)
    auto blocks_for = [&](int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, sm_count() * 16)); };
    cudaError_t e;
    const int64_t k_vals = c.kind == LISA_CACHE_SHARED && n_new < kTilePos ? rows * c.r : 0;
    if (c.dtype == LISA_BF16) e = launch_chained(append_kernel<uint4, 8, __nv_bfloat16>, dim3(blocks_for(std::max(rows * (c.d / 8), k_vals)), 2), dim3(threads), 0, s, p);
    else e = launch_chained(append_kernel<float4, 4, float>, dim3(blocks_for(std::max(rows * (c.d / 4), k_vals)), 2), dim3(threads), 0, s, p);
    count_launches(1);
    return e;
}

}  // namespace lisa
