// Projection GEMM on tcgen05 tensor cores: C[B*N, n_out] = X[B*N, K] . W[K, n_out], bf16 in, fp32 accumulation in tensor
// memory, bf16 out, the columns of C scattered straight into up to four [B, N, H, x] tensors (Eq. 1: H W^V_i and the
// product with W^O; Eq. 3: H W^Q_LR, H W^K_LR).
//
// One persistent CTA per SM walks 128 x 256 output tiles.  Warp 0 streams 64-deep K slices of X (K-major rows) and W
// (rows of n_out, i.e. the N dimension contiguous: an MN-major B operand, so W is used as stored, no transposed copy)
// through a four-stage TMA ring; warp 1 issues the MMAs (M 128, N 256, K 16) into one of two 256-column accumulators;
// warps 4-7 drain the other one (thread = output row), round to bf16 and store.  Every wait is bounded.
//
// Few rows (a decode step's projections: one row per sequence) are bound by streaming W once, which that split cannot do: 128-row
// tiles hold mostly padding and n_out / 256 of them leave most SMs without work.  tc_project_narrow_kernel turns the product
// round: the output columns are the M dimension (128 per CTA, W^T read as an MN-major A operand, again as stored), the rows
// -- all batches flattened -- the N dimension (16 to 256), and K is split over the CTAs of a cluster, which add their fp32
// partial sums through distributed shared memory.
#include <algorithm>

#include "common.cuh"
#include "tc_common.cuh"

namespace lisa {
namespace {

using namespace tc;

constexpr int BM = 128, BN = 256, BK = 64, STAGES = 4;
constexpr int A_BYTES = BM * BK * 2, B_BYTES = BK * BN * 2, STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int kThreads = 256;
constexpr int kMaxOut = 4;

struct ProjOut {
    void* ptr;
    int64_t sb, sn, sh;
    int32_t x, col0, cols;   // head width; first column of C and number of columns (H * x) that belong to this tensor
    int32_t row_dense;       // sh == x: a row's columns are contiguous from ptr + b*sb + n*sn
};

struct ProjParams {
    int B, N, K, n_out, n_outputs;
    int rows_per_batch;   // tiled rows per batch: N, or B * N with the batches flattened into one (tiled B is then 1)
    int tiled_b;
    int m_tiles_per_batch, n_tiles;
    long long tiles_total;
    ProjOut out[kMaxOut];
    int* status;
};

// Eight consecutive columns of C, from column `col` on, of row (b, n): one 16-byte store where the tensor that holds them
// allows it, else element by element (they may span two tensors or two heads).
__device__ __forceinline__ void store_columns(const ProjParams& p, int b, int n, int col, const uint4& v) {
    int o = 0;
    while (o + 1 < p.n_outputs && col >= p.out[o].col0 + p.out[o].cols) ++o;
    const ProjOut& t = p.out[o];
    const int rel = col - t.col0;
    __nv_bfloat16* base = reinterpret_cast<__nv_bfloat16*>(t.ptr) + b * t.sb + (int64_t)n * t.sn;
    if (t.row_dense && rel + 8 <= t.cols && ((reinterpret_cast<uintptr_t>(base + rel) & 15u) == 0)) {
        *reinterpret_cast<uint4*>(base + rel) = v;
        return;
    }
    const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(&v);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int cj = col + j;
        if (cj >= p.n_out) break;
        while (o + 1 < p.n_outputs && cj >= p.out[o].col0 + p.out[o].cols) ++o;
        const ProjOut& tt = p.out[o];
        const int rj = cj - tt.col0;
        reinterpret_cast<__nv_bfloat16*>(tt.ptr)[b * tt.sb + (int64_t)n * tt.sn + (int64_t)(rj / tt.x) * tt.sh + rj % tt.x] = e[j];
    }
}

constexpr int OFF_BAR = STAGES * STAGE_BYTES;
constexpr int SMEM_TOTAL = OFF_BAR + 256;

__global__ void __launch_bounds__(kThreads, 1)
tc_project_kernel(const __grid_constant__ ProjParams p, const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW) {
    extern __shared__ __align__(1024) uint8_t smem[];
    if ((smem_u32(smem) & 1023u) != 0) {
        if (threadIdx.x == 0) atomicAdd(p.status + 1, 1);
        return;
    }
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + OFF_BAR);
    uint64_t* full = bars;                 // [STAGES]
    uint64_t* empty = bars + STAGES;       // [STAGES]
    uint64_t* acc_full = bars + 2 * STAGES;    // [2]
    uint64_t* acc_empty = bars + 2 * STAGES + 2;   // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 4);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 2 * STAGES + 5);
    const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(acc_full + i, 1); mbar_init(acc_empty + i, 128); }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const int k_slices = (p.K + BK - 1) / BK;
    // tile index -> (batch, row tile, column tile); column tiles vary fastest so that concurrent CTAs share their X rows in L2
    auto tile_coord = [&](long long tile, int& b, int& mt, int& nt) {
        nt = (int)(tile % p.n_tiles);
        const long long r = tile / p.n_tiles;
        mt = (int)(r % p.m_tiles_per_batch);
        b = (int)(r / p.m_tiles_per_batch);
    };

    if (warp == 0) {
        // ------------------------------ TMA producer ------------------------------
        if (lane == 0) { tma_prefetch_desc(&tmX); tma_prefetch_desc(&tmW); }
        long long it = 0;   // running slice count over all tiles of this CTA
        bool ok = true;
        for (long long tile = blockIdx.x; ok && tile < p.tiles_total; tile += gridDim.x) {
            int b, mt, nt;
            tile_coord(tile, b, mt, nt);
            for (int ks = 0; ks < k_slices; ++ks, ++it) {
                const int s = (int)(it % STAGES);
                ok = mbar_wait(empty + s, (uint32_t)((it / STAGES) & 1) ^ 1u, abort_flag);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                uint8_t* sa = smem + s * STAGE_BYTES;
                uint8_t* sb = sa + A_BYTES;
                // X slice: [128 rows][64 k]; W slice: four [64 k][64 n] quarters
                if (elect_one()) {
                    mbar_expect_tx(full + s, STAGE_BYTES);
                    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
                                 ::"r"(smem_u32(sa)), "l"(&tmX), "r"(smem_u32(full + s)), "r"(ks * BK), "r"(mt * BM), "r"(b) : "memory");
#pragma unroll
                    for (int i = 0; i < BN / 64; ++i)
                        asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                                     ::"r"(smem_u32(sb + i * (BK * 128))), "l"(&tmW), "r"(smem_u32(full + s)), "r"(nt * BN + i * 64), "r"(ks * BK) : "memory");
                }
                __syncwarp();
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer (warp-uniform control flow, one elected lane issues) ------------------------------
        constexpr uint32_t IDESC = umma_idesc_bf16(BM, BN, 0, 1);   // X: K contiguous; W: N contiguous
        auto desc_off = [](uint64_t d, uint32_t bytes) -> uint64_t { return (d & 0xffffffff00000000ull) | (uint32_t)((uint32_t)d + (bytes >> 4)); };
        const uint64_t da0 = umma_desc_sw128(smem_u32(smem), 16, 1024);
        const uint64_t db0 = umma_desc_sw128(smem_u32(smem + A_BYTES), BK * 128, 1024);
        long long it = 0;
        int n_acc = 0;
        bool ok = true;
        for (long long tile = blockIdx.x; ok && tile < p.tiles_total; tile += gridDim.x, ++n_acc) {
            const int a = n_acc & 1;
            ok = mbar_wait(acc_empty + a, (uint32_t)((n_acc >> 1) & 1) ^ 1u, abort_flag);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            tc_fence_after();
            const uint32_t dst = tmem_base + a * BN;
            for (int ks = 0; ks < k_slices; ++ks, ++it) {
                const int s = (int)(it % STAGES);
                ok = mbar_wait(full + s, (uint32_t)((it / STAGES) & 1), abort_flag);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                tc_fence_after();
                const uint64_t da = desc_off(da0, s * STAGE_BYTES), db = desc_off(db0, s * STAGE_BYTES);
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk) umma_ss(dst, desc_off(da, kk * 32), desc_off(db, kk * 2048), IDESC, (ks > 0) || (kk > 0));
                    umma_commit(empty + s);
                    if (ks + 1 == k_slices) umma_commit(acc_full + a);
                }
                __syncwarp();
            }
        }
    } else if (warp >= 4) {
        // ------------------------------ epilogue (thread = output row) ------------------------------
        const int row = tid - 128;
        const uint32_t lane_sel = (uint32_t)((warp - 4) * 32) << 16;
        int n_acc = 0;
        bool ok = true;
        for (long long tile = blockIdx.x; ok && tile < p.tiles_total; tile += gridDim.x, ++n_acc) {
            int b, mt, nt;
            tile_coord(tile, b, mt, nt);
            const int a = n_acc & 1;
            if (!(ok = mbar_wait(acc_full + a, (uint32_t)((n_acc >> 1) & 1), abort_flag))) break;
            tc_fence_after();
            int n = mt * BM + row;
            const bool row_ok = n < p.rows_per_batch;
            if (p.tiled_b == 1) { b = n / p.N; n -= b * p.N; }
#pragma unroll 1
            for (int c = 0; c < BN / 32; ++c) {
                uint32_t r[32];
                tmem_ld32(tmem_base + a * BN + lane_sel + c * 32, r);
                tmem_wait_ld();
                if (c == BN / 32 - 1) {   // the accumulator is in registers: hand it back before the stores
                    tc_fence_before();
                    mbar_arrive(acc_empty + a);
                }
                const int col_base = nt * BN + c * 32;
                if (!row_ok || col_base >= p.n_out) continue;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const int col = col_base + g * 8;
                    if (col >= p.n_out) break;
                    uint4 v;
                    v.x = pack_bf16(__uint_as_float(r[g * 8 + 0]), __uint_as_float(r[g * 8 + 1]));
                    v.y = pack_bf16(__uint_as_float(r[g * 8 + 2]), __uint_as_float(r[g * 8 + 3]));
                    v.z = pack_bf16(__uint_as_float(r[g * 8 + 4]), __uint_as_float(r[g * 8 + 5]));
                    v.w = pack_bf16(__uint_as_float(r[g * 8 + 6]), __uint_as_float(r[g * 8 + 7]));
                    store_columns(p, b, n, col, v);
                }
            }
        }
    }
    // ------------------------------ teardown ------------------------------
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (tid == 0) atomicAdd(p.status + 1, 1);
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000ll) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ---------------------------------------------------------------------------------------------
// Few rows: a C^T tile of 64 (up to 64 rows) or 128 columns x NR rows per cluster, K split over the cluster's CTAs.
// Bound by HBM: W is read once.  Two CTAs per SM hold about 100 KB of slices each in flight; 64-column tiles halve the fp32
// partial sums that a given number of CTAs has to exchange, and slices of 128 k keep the producer at one copy of W per
// ~600 cycles (with 64 it spent its time issuing copies: 13.1 instead of 10.4 us at 1 x 4096 x 4096).  W's first slices are asked
// into L2 before the wait for the preceding kernel of the stream (L2 is coherent: a W which that kernel is still writing is only
// prefetched in vain).  Measured back to back, against the persistent kernel: 1 x 4096 x 5440 10.8 us (W alone at the copy rate:
// 6.8) instead of 38.1, 32 x 4096 x 5440 (one row per sequence) 11.4 instead of 148, 64 x 5120 x 6800 18 instead of 429.
// ---------------------------------------------------------------------------------------------
template <int NR>
struct Narrow {
    static constexpr int BN_ = NR <= 64 ? 64 : 128;               // columns of C per cluster: the M dimension of its MMAs
    static constexpr int KS = NR <= 64 ? 128 : 64;                // depth of a slice
    static constexpr int W_BYTES = KS * BN_ * 2, X_BYTES = NR * KS * 2, STAGE = W_BYTES + X_BYTES;
    static constexpr int ST = NR <= 16 ? 5 : NR <= 32 ? 4 : NR <= 64 ? 3 : NR <= 128 ? 3 : 4;
    static constexpr int CTAS = NR <= 128 ? 2 : 1;                // per SM
    static constexpr int BAR = ST * STAGE;
    static constexpr int TOTAL = BAR + 256;
    static constexpr uint32_t TMEM = NR < 32 ? 32 : NR;
    static_assert(NR * BN_ * 4 <= ST * STAGE, "the fp32 partial tile reuses the stages");
    static_assert(TOTAL * CTAS <= 232448 - 1024 * CTAS, "shared memory of an SM");
};
constexpr int kNarrowThreads = 192;   // warps 0-3 epilogue, 4 producer, 5 MMA issuer

template <int NR>
__global__ void __launch_bounds__(kNarrowThreads, Narrow<NR>::CTAS)
tc_project_narrow_kernel(const __grid_constant__ ProjParams p, const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW) {
    using S = Narrow<NR>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S::BAR);
    uint64_t* full = bars;                  // [ST]
    uint64_t* empty = bars + S::ST;         // [ST]
    uint64_t* acc_full = bars + 2 * S::ST;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S::ST + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 2 * S::ST + 2);
    const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
    const int split = gridDim.x, rank = blockIdx.x;             // the cluster spans grid dimension x
    const int nt = blockIdx.y, rt = blockIdx.z;
    const int rows = p.rows_per_batch;
    const bool aligned = (smem_u32(smem) & 1023u) == 0;           // uniform over the grid; a false one reports and computes nothing
    const int k_all = (p.K + S::KS - 1) / S::KS;
    const int k_begin = (int)((long long)k_all * rank / split), k_end = (int)((long long)k_all * (rank + 1) / split);
    const int n_slices = k_end - k_begin;
    if (tid == 0) {
        for (int i = 0; i < S::ST; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 1); }
        mbar_init(acc_full, 1);
        *abort_flag = aligned ? 0 : 1;
        fence_barrier_init();
    }
    if (warp == 5) tmem_alloc(tmem_slot, S::TMEM);
    constexpr int WB = S::BN_ / 64;   // 64-column boxes of a slice of W
    if (warp == 4) {
        const int s = lane / WB, c = nt * S::BN_ + (lane % WB) * 64;
        if (s < min(n_slices, S::ST) && c < p.n_out)
            asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(&tmW), "r"(c), "r"((k_begin + s) * S::KS) : "memory");
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    chain_release();   // not before every CTA holds its tensor memory (see common.cuh)
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    chain_wait();
    bool have = false;   // epilogue warps: the accumulator holds the CTA's share
    if (warp == 4) {
        if (lane == 0) { tma_prefetch_desc(&tmX); tma_prefetch_desc(&tmW); }
        bool ok = aligned;
        for (int i = 0; ok && i < n_slices; ++i) {
            const int s = i % S::ST;
            ok = mbar_wait(empty + s, (uint32_t)((i / S::ST) & 1) ^ 1u, abort_flag);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            uint8_t* sw = smem + s * S::STAGE;
            const int k0 = (k_begin + i) * S::KS;
            if (elect_one()) {
                mbar_expect_tx(full + s, S::STAGE);
#pragma unroll
                for (int c = 0; c < WB; ++c)
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                                 ::"r"(smem_u32(sw + c * (S::KS * 128))), "l"(&tmW), "r"(smem_u32(full + s)), "r"(nt * S::BN_ + c * 64), "r"(k0) : "memory");
#pragma unroll
                for (int c = 0; c < S::KS / 64; ++c)
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                                 ::"r"(smem_u32(sw + S::W_BYTES + c * (NR * 128))), "l"(&tmX), "r"(smem_u32(full + s)), "r"(k0 + c * 64), "r"(rt * NR) : "memory");
            }
            __syncwarp();
        }
    } else if (warp == 5) {
        constexpr uint32_t IDESC = umma_idesc_bf16(S::BN_, NR, 1, 0);   // W^T: columns contiguous (MN-major); X: K contiguous
        auto desc_off = [](uint64_t d, uint32_t bytes) -> uint64_t { return (d & 0xffffffff00000000ull) | (uint32_t)((uint32_t)d + (bytes >> 4)); };
        const uint64_t da0 = umma_desc_sw128(smem_u32(smem), S::KS * 128, 1024);
        const uint64_t db0 = umma_desc_sw128(smem_u32(smem + S::W_BYTES), 16, 1024);
        bool ok = aligned;
        for (int i = 0; ok && i < n_slices; ++i) {
            const int s = i % S::ST;
            ok = mbar_wait(full + s, (uint32_t)((i / S::ST) & 1), abort_flag);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            tc_fence_after();
            const uint64_t da = desc_off(da0, s * S::STAGE), db = desc_off(db0, s * S::STAGE);
            if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < S::KS / 16; ++kk)
                    umma_ss(tmem_base, desc_off(da, kk * 2048), desc_off(db, (kk >> 2) * (NR * 128) + (kk & 3) * 32), IDESC, (i > 0) || (kk > 0));
                if (i + S::ST < n_slices) umma_commit(empty + s);
                if (i + 1 == n_slices) umma_commit(acc_full);
            }
            __syncwarp();
        }
    } else {
        // thread = column of the tile; fp32 partial tile [row][columns] over the drained stages.  Tensor-memory lane of a column:
        // the column itself with 128 of them; with 64, sixteen per warp's quarter
        const int mycol = S::BN_ == 128 ? tid : (lane < 16 ? warp * 16 + lane : -1);
        have = aligned && mbar_wait(acc_full, 0, abort_flag);
        if (have) {
            tc_fence_after();
            float* part = reinterpret_cast<float*>(smem);
            const uint32_t lane_sel = (uint32_t)(warp * 32) << 16;
#pragma unroll 1
            for (int c = 0; c < NR; c += 32) {
                uint32_t r[32];
                tmem_ld32(tmem_base + lane_sel + c, r);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (c + j < NR && mycol >= 0) part[(c + j) * S::BN_ + mycol] = __uint_as_float(r[j]);
            }
        }
    }
    tc_fence_before();
    __syncwarp();
    // all partial tiles of the cluster are in place (a CTA that gave up takes part in both barriers like any other)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (!*abort_flag) {
        // this CTA's share of the tile: groups of eight columns, dealt round the cluster
        const int live = min(NR, rows - rt * NR);
        const uint32_t local = smem_u32(smem);
        for (int e = rank * kNarrowThreads + tid; e < live * (S::BN_ / 8); e += split * kNarrowThreads) {
            const int r = e / (S::BN_ / 8), g = e % (S::BN_ / 8);
            const int col = nt * S::BN_ + g * 8;
            if (col >= p.n_out) continue;
            float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            for (int q = 0; q < split; ++q) {   // in rank order: the sum does not depend on which CTA forms it
                uint32_t addr;
                float4 lo, hi;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(local + (uint32_t)(r * S::BN_ + g * 8) * 4), "r"(q));
                asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(lo.x), "=f"(lo.y), "=f"(lo.z), "=f"(lo.w) : "r"(addr));
                asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(hi.x), "=f"(hi.y), "=f"(hi.z), "=f"(hi.w) : "r"(addr + 16));
                acc[0] += lo.x; acc[1] += lo.y; acc[2] += lo.z; acc[3] += lo.w;
                acc[4] += hi.x; acc[5] += hi.y; acc[6] += hi.z; acc[7] += hi.w;
            }
            uint4 v;
            v.x = pack_bf16(acc[0], acc[1]); v.y = pack_bf16(acc[2], acc[3]); v.z = pack_bf16(acc[4], acc[5]); v.w = pack_bf16(acc[6], acc[7]);
            const int row = rt * NR + r, b = row / p.N;
            store_columns(p, b, row - b * p.N, col, v);
        }
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // nobody leaves while a peer still reads its tile
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (*abort_flag) {
        if (tid == 0) atomicAdd(p.status + 1, 1);
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000ll) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 5) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, S::TMEM);
    }
}

// General path: one thread per output element, fp32 accumulation in the order of k; any dtype and stride.
struct GenOut { void* ptr; int64_t sb, sn, sh; int32_t dtype, x, col0, cols; };
struct GenParams {
    int B, N, K, n_out, n_outputs;
    TView x;
    const void* w;
    int w_dtype;
    GenOut out[kMaxOut];
};
__global__ void generic_project_kernel(const __grid_constant__ GenParams p) {
    const int64_t total = (int64_t)p.B * p.N * p.n_out;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int col = (int)(e % p.n_out);
        const int64_t r = e / p.n_out;
        const int n = (int)(r % p.N), b = (int)(r / p.N);
        float acc = 0.f;
        for (int k = 0; k < p.K; ++k)
            acc = fmaf(ld_elem(p.x.ptr, b * p.x.sb + (int64_t)n * p.x.sn + k, p.x.dtype), ld_elem(p.w, (int64_t)k * p.n_out + col, p.w_dtype), acc);
        int o = 0;
        while (o + 1 < p.n_outputs && col >= p.out[o].col0 + p.out[o].cols) ++o;
        const GenOut& t = p.out[o];
        const int rel = col - t.col0;
        st_elem(t.ptr, b * t.sb + (int64_t)n * t.sn + (int64_t)(rel / t.x) * t.sh + rel % t.x, t.dtype, acc);
    }
}

}  // namespace

cudaError_t launch_generic_project(const lisa_project_args& a, cudaStream_t stream) {
    GenParams p{};
    p.B = a.B; p.N = a.N; p.K = a.d_in; p.n_outputs = a.n_outputs;
    p.x = make_view(a.x); p.w = a.w; p.w_dtype = a.w_dtype;
    int col = 0;
    for (int o = 0; o < a.n_outputs; ++o) {
        const lisa_project_output& src = a.outputs[o];
        p.out[o] = GenOut{src.t.ptr, src.t.stride_b, src.t.stride_n, src.t.stride_h, src.t.dtype, src.x, col, src.H * src.x};
        col += src.H * src.x;
    }
    p.n_out = col;
    const int64_t total = (int64_t)a.B * a.N * col;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, (int64_t)sm_count() * 32));
    generic_project_kernel<<<blocks, 256, 0, stream>>>(p);
    count_launches(1);
    return cudaGetLastError();
}

bool tc_project_supported(const lisa_project_args& a) {
    if (a.x.dtype != LISA_BF16 || a.w_dtype != LISA_BF16) return false;
    if ((reinterpret_cast<uintptr_t>(a.x.ptr) & 15u) || (reinterpret_cast<uintptr_t>(a.w) & 15u)) return false;
    if (a.d_in % 8 != 0 || a.x.stride_n % 8 != 0 || a.x.stride_b % 8 != 0 || a.x.stride_n < a.d_in) return false;
    int n_out = 0;
    for (int o = 0; o < a.n_outputs; ++o) {
        if (a.outputs[o].t.dtype != LISA_BF16) return false;
        n_out += a.outputs[o].H * a.outputs[o].x;
    }
    return n_out % 8 == 0;   // rows of W must be whole 16-byte units for the tensor map
}

namespace {
template <int NR>
cudaError_t prepare_narrow() {   // the default carveout leaves room for one CTA per SM only
    return allow_smem(tc_project_narrow_kernel<NR>, Narrow<NR>::TOTAL, true);
}
template <int NR>
cudaError_t launch_narrow_nr(const ProjParams& p, int split, int n_tiles, int row_tiles, const CUtensorMap& tmX, const CUtensorMap& tmW, cudaStream_t s) {
    using S = Narrow<NR>;
    cudaError_t e = prepare_narrow<NR>();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(split, n_tiles, row_tiles); cfg.blockDim = dim3(kNarrowThreads); cfg.dynamicSmemBytes = S::TOTAL; cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = split; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, tc_project_narrow_kernel<NR>, p, tmX, tmW);
}

cudaError_t launch_narrow(const lisa_project_args& a, const ProjParams& p, int64_t row_stride, cudaStream_t stream) {
    const int rows = p.rows_per_batch;
    const int nr = rows <= 16 ? 16 : rows <= 32 ? 32 : rows <= 64 ? 64 : rows <= 128 ? 128 : 256;
    const int bn = nr <= 64 ? 64 : 128, ks = nr <= 64 ? 128 : 64;   // tile width and slice depth of the build (Narrow)
    const int n_tiles = (p.n_out + bn - 1) / bn, row_tiles = (rows + nr - 1) / nr, k_slices = (a.d_in + ks - 1) / ks;
    // K is split as far as all CTAs are resident at once, clusters included (7/8 of the slots: a cluster's CTAs share a GPC and
    // cannot fill every one of its SMs); a second, short wave costs more than the shorter K ranges save (1 x 4096 x 12288:
    // 20.5 us with one range, 25.9 with two).  At most 8 CTAs a cluster, two slices a CTA, and from 128 rows on a split of 4,
    // because the fp32 partial sums cross the SM-to-SM network once per CTA (128 x 4096 x 4096: 17.6 us at 4, 20.9 at 8).
    const int tiles = n_tiles * row_tiles, slots = nr <= 128 ? 2 * sm_count() * 7 / 8 : sm_count();
    const int split = std::max(1, std::min({nr <= 64 ? 8 : 4, slots / tiles, k_slices / 2}));
    CUtensorMap tmX, tmW;
    const uint64_t xd[2] = {(uint64_t)a.d_in, (uint64_t)rows}, xs[1] = {(uint64_t)row_stride * 2};
    const uint32_t xb[2] = {(uint32_t)BK, (uint32_t)nr};
    const uint64_t wd[2] = {(uint64_t)p.n_out, (uint64_t)a.d_in}, ws[1] = {(uint64_t)p.n_out * 2};
    const uint32_t wb[2] = {64, (uint32_t)ks};
    if (!make_tensor_map_bf16(&tmX, a.x.ptr, 2, xd, xs, xb) || !make_tensor_map_bf16(&tmW, a.w, 2, wd, ws, wb)) return cudaErrorInvalidValue;
    count_launches(1);
    switch (nr) {
        case 16: return launch_narrow_nr<16>(p, split, n_tiles, row_tiles, tmX, tmW, stream);
        case 32: return launch_narrow_nr<32>(p, split, n_tiles, row_tiles, tmX, tmW, stream);
        case 64: return launch_narrow_nr<64>(p, split, n_tiles, row_tiles, tmX, tmW, stream);
        case 128: return launch_narrow_nr<128>(p, split, n_tiles, row_tiles, tmX, tmW, stream);
        default: return launch_narrow_nr<256>(p, split, n_tiles, row_tiles, tmX, tmW, stream);
    }
}
}  // namespace

cudaError_t launch_tc_project(const lisa_project_args& a, cudaStream_t stream) {
    ProjParams p{};
    p.B = a.B; p.N = a.N; p.K = a.d_in; p.n_outputs = a.n_outputs;
    int col = 0;
    for (int o = 0; o < a.n_outputs; ++o) {
        const lisa_project_output& src = a.outputs[o];
        ProjOut& t = p.out[o];
        t.ptr = src.t.ptr; t.sb = src.t.stride_b; t.sn = src.t.stride_n; t.sh = src.t.stride_h;
        t.x = src.x; t.col0 = col; t.cols = src.H * src.x;
        t.row_dense = (src.t.stride_h == src.x || src.H == 1) ? 1 : 0;
        col += t.cols;
    }
    p.n_out = col;
    // Rows at one constant distance (a dense x, one sequence, or one row per sequence) are tiled as one long batch.
    int64_t row_stride = (a.N == 1 && a.B > 1) ? a.x.stride_b : a.x.stride_n;
    const bool flat = (a.B == 1 || a.N == 1 || a.x.stride_b == a.N * a.x.stride_n) && (int64_t)a.B * a.N <= 0x7fffffff && row_stride >= a.d_in;
    if (!flat) row_stride = a.x.stride_n;
    p.tiled_b = flat ? 1 : a.B;
    p.rows_per_batch = flat ? a.B * a.N : a.N;
    p.status = status_words();
    if (!p.status) return cudaErrorUnknown;
    // The narrow kernel as long as its CTAs fit the SMs; beyond, the persistent kernel's 256-column tiles fill them as well
    // (4096 x 5440, 512 rows: 37 us against 40; 4096 x 12288, 512 rows: 77 against 76, and 40 against 51 at 256 rows).
    // Its column tiles are a grid dimension of at most 65535.
    const int narrow_tiles = ((p.n_out + 127) / 128) * ((p.rows_per_batch + 255) / 256);
    if (flat && (p.n_out + 63) / 64 <= 65535 && (p.rows_per_batch <= 128 || (p.rows_per_batch <= 512 && narrow_tiles <= sm_count()))) return launch_narrow(a, p, row_stride, stream);
    p.m_tiles_per_batch = (p.rows_per_batch + BM - 1) / BM;
    p.n_tiles = (p.n_out + BN - 1) / BN;
    p.tiles_total = (long long)p.tiled_b * p.m_tiles_per_batch * p.n_tiles;
    CUtensorMap tmX, tmW;
    {
        const uint64_t dims[3] = {(uint64_t)a.d_in, (uint64_t)p.rows_per_batch, (uint64_t)p.tiled_b};
        const uint64_t str[2] = {(uint64_t)row_stride * 2, (uint64_t)(flat ? row_stride : a.x.stride_b) * 2};
        const uint32_t box[3] = {(uint32_t)BK, (uint32_t)BM, 1};
        if (!make_tensor_map_bf16(&tmX, a.x.ptr, 3, dims, str, box)) return cudaErrorInvalidValue;
    }
    {
        const uint64_t dims[2] = {(uint64_t)p.n_out, (uint64_t)a.d_in};
        const uint64_t str[1] = {(uint64_t)p.n_out * 2};
        const uint32_t box[2] = {64, (uint32_t)BK};
        if (!make_tensor_map_bf16(&tmW, a.w, 2, dims, str, box)) return cudaErrorInvalidValue;
    }
    cudaError_t e;
    if ((e = allow_smem(tc_project_kernel, SMEM_TOTAL)) != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::min<long long>(p.tiles_total, sm_count());
    tc_project_kernel<<<grid, kThreads, SMEM_TOTAL, stream>>>(p, tmX, tmW);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace lisa
