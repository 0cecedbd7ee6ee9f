// Head-axis aligner (Sec. 5.1), one link per launch, on tcgen05: single links of prompts above one wave, and the shapes and Integrate
// modes the chain kernel of tc_align.cu does not take:
//   CONCAT  (32 heads)        A_k = W2^T act(W1^T [A_{k-1}; D_k] + b1) + b2    W1 [64, m], W2 [m, 32], m <= 256: the paper's
//                             complete model (Sec. 5.1, "An overview of LiSA": 64 x 256 and 256 x 32), and its one-layer
//                             form A_k = W1^T [A_{k-1}; D_k] + b1 with W1 [64, 32]
//   ADD     (32 or 40 heads)  A_k = FFN_k(A_{k-1}) + D_k with a two-layer FFN of hidden width m <= 256 (40 -> 80 -> 40 is the
//                             LLaMA2-13B shape), one linear layer, or no FFN at all (PLUS)
// Forms without a hidden layer run with an identity first layer (exact: every hidden unit is one fp16 input times one).
//
// Planes (fp16, blocked [row block of 128][column block of 64][row][B*heads + head][64 columns]):
//   plane_x  the link's input scores (A_0 = Q0.K0^T/sqrt(d) for the first link)
//   plane_d  D_k = Q'_k.K'_k^T/sqrt(r), already scaled (Eq. 3); ADD: may be absent (the top link's difference is added by
//            the attention kernel)
// Outputs go over the inputs, which are dead once the launch has read them: the scores for the next link (unscaled) and
// log2(e) times the FFN output for the attention kernel (which works in the exp2 domain), each over plane_x or plane_d
// as the caller says.
//
// A tile is 64 key positions of two query rows: 128 positions, the M of both MMAs.  In a plane the positions of a head are
// 128 contiguous bytes, so the TMA-loaded tile is the first layer's A operand as it stands (M-major, K = heads); its fp32
// result goes from tensor memory through the registers (bias, activation, rounding to fp16) back into tensor memory, where
// it is the second layer's A operand.  Nothing but the planes and the weights (B operands, in shared memory for the whole
// launch) touches shared memory.  Roles: one warp loads, one issues each layer's MMAs, and BUFS tiles are in flight, each with
// 512 / BUFS columns of tensor memory, so that the waits of one tile (two MMAs, four barriers) hide behind the arithmetic of
// the others.  There are always four warpgroups: with two tiles in flight, two share a tile, half of the hidden layer and half
// of the heads each.
// Measured: 64 -> 256 -> 32 on 2048 tokens of 32 heads 272 us with warp-level MMAs (their fragments came through shared
// memory), 120 us now, where the planes' 415 MB take 63; 40 -> 80 -> 40 on 2 x 1777 tokens 138 us before, 97 now (80).
#include <algorithm>

#include "tc_align_mma.cuh"

namespace lisa {
namespace {

using namespace tc;
using alignmma::act_h2;
using alignmma::KIND_FFN;
using alignmma::KIND_PLUS;
using alignmma::KIND_SINGLE;
using alignmma::kLog2e;
using alignmma::ldmatrix_x4_trans;
using alignmma::ldw;
using alignmma::stmatrix_x4_trans;

constexpr int UNIT = 128;
constexpr int kMaxStages = 8;

struct LinkParams {
    int N, row0, d_row0;                // first query row of plane_x / plane_d
    int row_begin, row_end;             // query rows of the launch
    int tiles_per_batch, total;         // tiles: (row pair, 64-column block up to the diagonal)
    int has_d;                          // a difference plane is read (always with CONCAT)
    int dst_next, dst_scaled;           // where the next link's input / the attention kernel's plane go: -1 nowhere, 0 plane_x, 1 plane_d
    const void *w1, *b1, *w2, *b2;
    int w_dtype, m, kind;               // kind: KIND_FFN (hidden width m) / KIND_SINGLE / KIND_PLUS
    int hid;                            // hidden units of the MMAs: m (or the inputs, without a hidden layer) rounded up to 16
    int stages;
    int* status;
};

// Shared memory of a launch: [stages][plane x, plane d][2 rows][heads][128 B], zero rows, weights, staging, biases, barriers.
template <int NH, bool CONCAT, int BUFS>
struct Shape {
    static constexpr int HK = (NH + 15) / 16 * 16;            // heads as an MMA's K (or N): zero-padded to 16
    static constexpr int H_IN = CONCAT ? 2 * NH : NH;
    static constexpr int K1 = CONCAT ? 2 * HK : HK;
    static constexpr int SLOT = NH * 128;                     // one query row of a tile
    static constexpr int TILE = 2 * SLOT;
    static constexpr int ZERO = HK == NH ? 0 : SLOT + 1024;   // the padding heads of both rows (see the first layer's issuer)
    static constexpr int TW = 4 / BUFS;                       // warpgroups that share a tile
    static constexpr int STRIDE = 512 / BUFS;                 // tensor-memory columns of a tile in flight
    // Hidden units HALF * i .. of warpgroup i of a tile.  Their sums are read from columns HALF * i and written back, half as wide, from
    // the same column on, so that the two never touch what the other has not read; the second layer's result follows the first's.
    static constexpr int HALF = STRIDE / TW, D_OFF = HALF / 2;
    static constexpr int NG = NH / 8, GW = (NG + TW - 1) / TW;   // groups of 8 heads; of a warpgroup
    static constexpr int BOX = NG % TW == 0 ? GW * 8 : 8;     // heads of one copy out
    static constexpr int STG = GW * 8 * 64;                   // a warp's 32 positions of its heads on the way out
    static constexpr int CHUNK = 32;                          // hidden units a thread holds at a time (registers)
    static constexpr int THREADS = 4 * 128 + 96;              // + loader, two MMA issuers
    static_assert(K1 <= 64 && (!CONCAT || HK == NH) && D_OFF + HK <= HALF, "layout");
    static __host__ __device__ int stage_bytes(bool has_d) { return TILE * (has_d ? 2 : 1); }
    static __host__ __device__ int w1_off(int stages, bool has_d) { return stages * stage_bytes(has_d) + ZERO; }
    static __host__ __device__ int w2_off(int w1, int hid) { return w1 + hid * 128; }
    static __host__ __device__ int stg_off(int w2, int hid) { return w2 + (hid + 63) / 64 * (HK * 128); }
    static __host__ __device__ int bias_off(int stg) { return stg + 16 * 2 * STG; }
    static __host__ __device__ int bar_off(int bias, int hid) { return bias + hid * 2 + HK * 4; }
    static __host__ int total(int stages, bool has_d, int hid) {
        return bar_off(bias_off(stg_off(w2_off(w1_off(stages, has_d), hid), hid)), hid) + (2 * kMaxStages + 4 * 4) * 8 + 16;
    }
};

__host__ __device__ constexpr uint32_t umma_idesc_f16(int M, int N, int a_mn_major, int b_mn_major) {
    return (1u << 4) | ((uint32_t)a_mn_major << 15) | ((uint32_t)b_mn_major << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}

// 16 lanes x 8 columns as an MMA accumulator fragment: thread t gets columns 2(t % 4), + 1 of lanes t / 4 and t / 4 + 8
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, float* r) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];" : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void stmatrix_x2_trans(uint32_t saddr, uint32_t r0, uint32_t r1) {
    asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1,%2};" ::"r"(saddr), "r"(r0), "r"(r1) : "memory");
}
// A warp's results, times `scale`, as [head][32 positions] rows of 64 bytes whose 16-byte chunks carry the copy engine's 64-byte swizzle.
template <int NG>
__device__ __forceinline__ void put_frags(uint32_t stg, int lane, const float (*y)[NG][4], float scale) {
#pragma unroll
    for (int s2 = 0; s2 < 2; ++s2)
#pragma unroll
        for (int g = 0; g < NG; g += 2) {
            const int head = (g + (lane >> 4)) * 8 + (lane & 7), chunk = 2 * s2 + ((lane >> 3) & 1);   // x2 reads lanes 0-15 only
            const uint32_t addr = stg + head * 64 + ((chunk ^ ((head >> 1) & 3)) << 4);
            uint32_t r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float* v = y[s2][min(g + (k >> 1), NG - 1)] + 2 * (k & 1);
                r[k] = pack_f16(v[0] * scale, v[1] * scale);
            }
            if (g + 1 < NG) stmatrix_x4_trans(addr, r);
            else stmatrix_x2_trans(addr, r[0], r[1]);
        }
}

// Two hidden units: the MMA's sums rounded to fp16, plus the bias, through the activation.
template <int ACT>
__device__ __forceinline__ uint32_t hidden_pair(float lo, float hi, uint32_t bias) {
    const uint32_t x = pack_f16(lo, hi);
    uint32_t r;
    if constexpr (ACT == LISA_ACT_RELU) {
        asm("fma.rn.relu.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(0x3c003c00u), "r"(bias));
        return r;
    } else {
        asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(bias));
        return act_h2<ACT>(r);
    }
}

// Position of a tile in the launch: (sequence, first of two query rows, 64-column block)
struct Cursor {
    int b, r, jb;
    __device__ __forceinline__ void seek(const LinkParams& p, int t) {
        b = t / p.tiles_per_batch;
        int rem = t - b * p.tiles_per_batch;
        r = p.row_begin;
        for (;;) {   // blocks of 64 query rows
            const int pairs = (min(p.row_end - r, 64) + 1) / 2, cols = (r >> 6) + 1;
            if (rem < pairs * cols) {
                r += rem / cols * 2;
                jb = rem % cols;
                return;
            }
            rem -= pairs * cols;
            r += 64;
        }
    }
    __device__ __forceinline__ void step(const LinkParams& p) {
        if (++jb <= (r >> 6)) return;
        jb = 0;
        if ((r += 2) < p.row_end) return;
        r = p.row_begin;
        ++b;
    }
};

template <int NH, bool CONCAT, int ACT, int BUFS>
__global__ void __launch_bounds__(Shape<NH, CONCAT, BUFS>::THREADS, 1)
tc_align_link_kernel(const __grid_constant__ LinkParams p, const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmD,
                     const __grid_constant__ CUtensorMap tmXs, const __grid_constant__ CUtensorMap tmDs) {
    using S = Shape<NH, CONCAT, BUFS>;
    constexpr int HK = S::HK, K1 = S::K1, SLOT = S::SLOT, TILE = S::TILE, STG = S::STG;
    extern __shared__ __align__(1024) uint8_t smem[];
    if ((smem_u32(smem) & 1023u) != 0) {   // the swizzled tiles' bases: refuse loudly instead of computing garbage
        if (threadIdx.x == 0) atomicAdd(p.status + 1, 1);
        return;
    }
    const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
    const int hid = p.hid, stages = p.stages, kind = p.kind, m = p.m, wd = p.w_dtype;
    const bool has_d = p.has_d != 0;
    const int stage_bytes = S::stage_bytes(has_d);
    const int w1_off = S::w1_off(stages, has_d), w2_off = S::w2_off(w1_off, hid), stg_off = S::stg_off(w2_off, hid);
    const int bias_off = S::bias_off(stg_off), bar_off = S::bar_off(bias_off, hid);
    uint8_t* sW1 = smem + w1_off;                                      // [hidden][64 inputs], swizzled
    uint8_t* sW2 = smem + w2_off;                                      // [64 hidden units][heads, padded][64], swizzled
    uint32_t* b1h = reinterpret_cast<uint32_t*>(smem + bias_off);      // [hid / 2] packed fp16 pairs
    float* b2 = reinterpret_cast<float*>(b1h + hid / 2);               // [HK]
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + bar_off);
    uint64_t* full = bars;                       // [stages]
    uint64_t* empty = bars + kMaxStages;         // [stages] first layer done (and, where it is added later, plane d read)
    uint64_t* s_full = bars + 2 * kMaxStages;    // [BUFS] first layer's sums
    uint64_t* h_full = s_full + 4;               // [BUFS] hidden layer written back
    uint64_t* o_full = s_full + 8;               // [BUFS] second layer's sums
    uint64_t* b_free = s_full + 12;              // [BUFS] ... read: the columns are free
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_full + 16);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    // this CTA's contiguous range of tiles
    const int per = (p.total + (int)gridDim.x - 1) / (int)gridDim.x;
    const int t_begin = min(p.total, (int)blockIdx.x * per), n_tiles = min(p.total, t_begin + per) - t_begin;

    // barriers and tensor memory are set up under the tail of the kernel before this one; not the weights, which it may have written
    for (int e = tid; e < S::ZERO / 16; e += S::THREADS)
        *reinterpret_cast<uint4*>(smem + stages * stage_bytes + e * 16) = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
        for (int i = 0; i < stages; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, (!CONCAT && has_d) ? 1 + 4 * S::TW : 1); }
        for (int i = 0; i < BUFS; ++i) { mbar_init(s_full + i, 1); mbar_init(h_full + i, 4 * S::TW); mbar_init(o_full + i, 1); mbar_init(b_free + i, 4 * S::TW); }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 0) tmem_alloc(tmem_slot, 512);
    if (warp == 16 && elect_one()) {
        tma_prefetch_desc(&tmX); tma_prefetch_desc(&tmXs);
        if (has_d) { tma_prefetch_desc(&tmD); tma_prefetch_desc(&tmDs); }
    }
    __syncwarp();
    chain_wait();

    // ---- weights as fp16 B operands; inputs beyond the heads and hidden units beyond m are zero ----
    auto first = [&](int k, int n) -> float {      // [inputs][hidden]
        if (k >= S::H_IN) return 0.f;
        if (kind != KIND_FFN) return k == n ? 1.f : 0.f;
        return n < m ? ld_elem(p.w1, k * m + n, wd) : 0.f;
    };
    auto second = [&](int k, int n) -> float {     // [hidden][heads]
        if (n >= NH) return 0.f;
        if (kind == KIND_FFN) return k < m ? ld_elem(p.w2, k * NH + n, wd) : 0.f;
        if (kind == KIND_SINGLE) return k < S::H_IN ? ld_elem(p.w1, k * NH + n, wd) : 0.f;
        return k == n ? 1.f : 0.f;
    };
    for (int e = tid; e < hid * (K1 / 8); e += S::THREADS) {
        const int n = e % hid, k = e / hid * 8;
        uint4 v;
        v.x = pack_f16(first(k, n), first(k + 1, n)); v.y = pack_f16(first(k + 2, n), first(k + 3, n));
        v.z = pack_f16(first(k + 4, n), first(k + 5, n)); v.w = pack_f16(first(k + 6, n), first(k + 7, n));
        *reinterpret_cast<uint4*>(sW1 + sw128_offset(n, k >> 3)) = v;
    }
    for (int e = tid; e < HK * (hid / 8); e += S::THREADS) {
        const int n = e % HK, k = e / HK * 8;
        uint4 v;
        v.x = pack_f16(second(k, n), second(k + 1, n)); v.y = pack_f16(second(k + 2, n), second(k + 3, n));
        v.z = pack_f16(second(k + 4, n), second(k + 5, n)); v.w = pack_f16(second(k + 6, n), second(k + 7, n));
        *reinterpret_cast<uint4*>(sW2 + (k >> 6) * (HK * 128) + sw128_offset(n, (k >> 3) & 7)) = v;
    }
    for (int e = tid; e < hid / 2; e += S::THREADS)
        b1h[e] = (kind != KIND_FFN || 2 * e >= m) ? 0u : pack_f16(ldw(p.b1, 2 * e, wd), 2 * e + 1 < m ? ldw(p.b1, 2 * e + 1, wd) : 0.f);
    for (int e = tid; e < HK; e += S::THREADS)
        b2[e] = e >= NH ? 0.f : (kind == KIND_FFN ? ldw(p.b2, e, wd) : (kind == KIND_SINGLE ? ldw(p.b1, e, wd) : 0.f));
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    chain_release();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);

    if (warp == 16) {
        // ------------------------------ loader: one thread, one copy per plane and tile ------------------------------
        // (a copy per query row, issued by two lanes of a converged warp, took 1300 cycles a tile: more than the tile's arithmetic)
        if (elect_one()) {
            Cursor cu;
            if (n_tiles > 0) cu.seek(p, t_begin);
            int s = 0;
            uint32_t par = 1;
            for (int i = 0; i < n_tiles; ++i) {
                if (!mbar_wait(empty + s, par, abort_flag)) break;
                mbar_expect_tx(full + s, (has_d ? 2 : 1) * TILE);
                uint8_t* dst = smem + s * stage_bytes;
                const int rx = cu.r - p.row0, rd = cu.r - p.d_row0;
                tma_load_5d(dst, &tmX, full + s, 0, cu.b * NH, rx & 127, cu.jb, rx >> 7);
                if (has_d) tma_load_5d(dst + TILE, &tmD, full + s, 0, cu.b * NH, rd & 127, cu.jb, rd >> 7);
                cu.step(p);
                if (++s == stages) { s = 0; par ^= 1; }
            }
        }
        __syncwarp();
    } else if (warp == 17) {
        // ------------------------------ MMA issuer: first layer ------------------------------
        const uint32_t idesc = umma_idesc_f16(128, hid, 1, 0);
        const uint64_t db0 = umma_desc_sw128(smem_u32(sW1), 16, 1024);
        auto desc_off = [](uint64_t d, uint32_t bytes) -> uint64_t { return (d & 0xffffffff00000000ull) | (uint32_t)((uint32_t)d + (bytes >> 4)); };
        int s = 0, w = 0;
        uint32_t par = 0, wpar = 1;
        for (int i = 0; i < n_tiles; ++i) {
            bool ok = mbar_wait(full + s, par, abort_flag) && mbar_wait(b_free + w, wpar, abort_flag);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t st = smem_u32(smem) + s * stage_bytes;
                const uint64_t da = umma_desc_sw128(st, SLOT, 1024);
#pragma unroll
                for (int ks = 0; ks < K1 / 16; ++ks) {   // 16 heads = two groups of 8 rows; the second half of K lies in plane d's tile
                    const uint32_t a_off = ks < HK / 16 ? ks * 2048 : TILE + (ks - HK / 16) * 2048;
                    uint64_t a = desc_off(da, a_off);
                    // 40 heads: the last group's partner is eight zero rows behind the stages (for the tile's second row SLOT further on)
                    if (HK != NH && ks == HK / 16 - 1) a = umma_desc_sw128(st + a_off, SLOT, smem_u32(smem) + stages * stage_bytes - (st + a_off));
                    umma_ss(tmem_base + w * S::STRIDE, a, desc_off(db0, ks * 32), idesc, ks > 0);
                }
                umma_commit(empty + s);
                umma_commit(s_full + w);
            }
            __syncwarp();
            if (++s == stages) { s = 0; par ^= 1; }
            if (++w == BUFS) { w = 0; wpar ^= 1; }
        }
    } else if (warp == 18) {
        // ------------------------------ MMA issuer: second layer ------------------------------
        constexpr uint32_t idesc = umma_idesc_f16(128, HK, 0, 0);
        const uint64_t db0 = umma_desc_sw128(smem_u32(sW2), 16, 1024);
        auto desc_off = [](uint64_t d, uint32_t bytes) -> uint64_t { return (d & 0xffffffff00000000ull) | (uint32_t)((uint32_t)d + (bytes >> 4)); };
        int w = 0;
        uint32_t wpar = 0;
        for (int i = 0; i < n_tiles; ++i) {
            bool ok = mbar_wait(h_full + w, wpar, abort_flag);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            tc_fence_after();
            const uint32_t buf = tmem_base + w * S::STRIDE;
            if (elect_one()) {
#pragma unroll
                for (int i2 = 0; i2 < S::TW; ++i2) {
                    const int n_ks = min(hid - i2 * S::HALF, S::HALF) / 16;   // k-steps of this warpgroup's hidden units
                    const uint32_t a = buf + i2 * S::HALF, b_ks = i2 * (S::HALF / 16);
                    int ks = 0;
                    for (; ks + 4 <= n_ks; ks += 4) {
                        const uint64_t db = desc_off(db0, ((b_ks + ks) >> 2) * (HK * 128));
#pragma unroll
                        for (int k = 0; k < 4; ++k) umma_ts(buf + S::D_OFF, a + (ks + k) * 8, desc_off(db, k * 32), idesc, b_ks + ks + k > 0);
                    }
                    for (; ks < n_ks; ++ks)
                        umma_ts(buf + S::D_OFF, a + ks * 8, desc_off(db0, ((b_ks + ks) >> 2) * (HK * 128) + (ks & 3) * 32), idesc, b_ks + ks > 0);
                }
                umma_commit(o_full + w);
            }
            __syncwarp();
            if (++w == BUFS) { w = 0; wpar ^= 1; }
        }
    } else {
        // ------------------------------ warpgroups: hidden layer and results (thread = position) ------------------------------
        const int w = (warp >> 2) / S::TW, hf = (warp >> 2) % S::TW, q = warp & 3;   // tile in flight, share of it, quarter of the positions
        const uint32_t buf = tmem_base + w * S::STRIDE + ((uint32_t)(q * 32) << 16);
        const int dst_next = p.dst_next, dst_scaled = p.dst_scaled;
        uint8_t* stg = smem + stg_off + warp * (2 * STG);
        const uint32_t stg_u32 = smem_u32(stg);
        constexpr int NG = S::NG, GW = S::GW;
        const int g0 = hf * GW;   // this warpgroup's first group of heads; groups beyond the last are computed as the last and not stored
        float2 bias2[GW];
#pragma unroll
        for (int g = 0; g < GW; ++g) bias2[g] = *reinterpret_cast<const float2*>(b2 + min(g0 + g, NG - 1) * 8 + 2 * (lane & 3));
        Cursor cu;
        if (w < n_tiles) cu.seek(p, t_begin + w);
        int s = w % stages;
        uint32_t spar = (w / stages) & 1, wpar = 0;
        for (int i = w; i < n_tiles; i += BUFS) {
            if (!__all_sync(0xffffffffu, mbar_wait(s_full + w, wpar, abort_flag))) break;
            tc_fence_after();
            const uint32_t col = buf + hf * S::HALF;
            const uint32_t* bias1 = b1h + hf * (S::HALF / 2);
            const int units = min(hid - hf * S::HALF, S::HALF);
            int c = 0;
            for (; c + S::CHUNK <= units; c += S::CHUNK) {
                uint32_t f[S::CHUNK], h[S::CHUNK / 2];
#pragma unroll
                for (int k = 0; k < S::CHUNK; k += 32) tmem_ld32(col + c + k, f + k);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < S::CHUNK / 8; ++j) {
                    const uint4 bb = *reinterpret_cast<const uint4*>(bias1 + c / 2 + 4 * j);
                    h[4 * j + 0] = hidden_pair<ACT>(__uint_as_float(f[8 * j + 0]), __uint_as_float(f[8 * j + 1]), bb.x);
                    h[4 * j + 1] = hidden_pair<ACT>(__uint_as_float(f[8 * j + 2]), __uint_as_float(f[8 * j + 3]), bb.y);
                    h[4 * j + 2] = hidden_pair<ACT>(__uint_as_float(f[8 * j + 4]), __uint_as_float(f[8 * j + 5]), bb.z);
                    h[4 * j + 3] = hidden_pair<ACT>(__uint_as_float(f[8 * j + 6]), __uint_as_float(f[8 * j + 7]), bb.w);
                }
#pragma unroll
                for (int k = 0; k < S::CHUNK / 2; k += 16) tmem_st16(col + c / 2 + k, h + k);
            }
            for (; c < units; c += 16) {
                uint32_t f[16], h[8];
                tmem_ld16(col + c, f);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 8; ++j) h[j] = hidden_pair<ACT>(__uint_as_float(f[2 * j]), __uint_as_float(f[2 * j + 1]), bias1[c / 2 + j]);
                tmem_st8(col + c / 2, h);
            }
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(h_full + w);

            if (!__all_sync(0xffffffffu, mbar_wait(o_full + w, wpar, abort_flag))) break;
            wpar ^= 1;
            tc_fence_after();
            // a warp's 32 positions as two strips of 16, eight heads at a time: lane holds heads 2(lane % 4), + 1 of positions lane / 4, + 8,
            // the fragment arrangement stmatrix and ldmatrix transpose from and to [head][position] rows
            float y[2][GW][4];
#pragma unroll
            for (int s2 = 0; s2 < 2; ++s2)
#pragma unroll
                for (int g = 0; g < GW; ++g) tmem_ld_frag(buf + S::D_OFF + ((uint32_t)(s2 * 16) << 16) + min(g0 + g, NG - 1) * 8, y[s2][g]);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (elect_one()) {
                mbar_arrive(b_free + w);
                tma_store_wait_read<0>();   // the previous tile's stores have read the staging buffers
            }
            __syncwarp();
#pragma unroll
            for (int s2 = 0; s2 < 2; ++s2)
#pragma unroll
                for (int g = 0; g < GW; ++g) {
                    y[s2][g][0] += bias2[g].x; y[s2][g][1] += bias2[g].y;
                    y[s2][g][2] += bias2[g].x; y[s2][g][3] += bias2[g].y;
                }
            if (dst_scaled >= 0) put_frags<GW>(stg_u32, lane, y, kLog2e);
            if (!CONCAT && has_d) {   // A_k = FFN(A_{k-1}) + D_k
                if (!__all_sync(0xffffffffu, mbar_wait(full + s, spar, abort_flag))) break;
                const uint32_t db = smem_u32(smem) + s * stage_bytes + TILE + (q >> 1) * SLOT;
#pragma unroll
                for (int s2 = 0; s2 < 2; ++s2)
#pragma unroll
                    for (int g = 0; g < GW; g += 2) {
                        // four 8 x 8 blocks: (heads g, positions 0-7), (g, 8-15), (g + 1, 0-7), (g + 1, 8-15); beyond the last head: g again
                        const int head = min(g0 + g + (lane >> 4), NG - 1) * 8 + (lane & 7), chunk = (q & 1) * 4 + 2 * s2 + ((lane >> 3) & 1);
                        uint32_t dfr[4];
                        ldmatrix_x4_trans(dfr, db + sw128_offset(head, chunk));
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (g + (k >> 1) >= GW) break;
                            const float2 dv = unpack_f16(dfr[k]);
                            y[s2][g + (k >> 1)][2 * (k & 1)] += dv.x;
                            y[s2][g + (k >> 1)][2 * (k & 1) + 1] += dv.y;
                        }
                    }
                __syncwarp();
                if (lane == 0) mbar_arrive(empty + s);
            }
            if (dst_next >= 0) put_frags<GW>(stg_u32 + STG, lane, y, 1.f);
            fence_async_smem();
            __syncwarp();
            if (elect_one()) {
                const int row = cu.r + (q >> 1), x = (q & 1) * 32;
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int rel = row - (k ? p.d_row0 : p.row0);
                    const CUtensorMap* map = k ? &tmDs : &tmXs;
#pragma unroll
                    for (int g = 0; g < GW; g += S::BOX / 8) {
                        if (g0 + g >= NG) break;
                        const int head = cu.b * NH + (g0 + g) * 8;
                        if (dst_scaled == k) tma_store_5d(map, stg + g * 512, x, head, rel & 127, cu.jb, rel >> 7);
                        if (dst_next == k) tma_store_5d(map, stg + STG + g * 512, x, head, rel & 127, cu.jb, rel >> 7);
                    }
                }
                tma_store_commit();
            }
#pragma unroll
            for (int k = 0; k < BUFS; ++k) {
                cu.step(p);
                if (++s == stages) { s = 0; spar ^= 1; }
            }
        }
        if (elect_one()) tma_store_wait_all<0>();
        __syncwarp();
    }
    // ------------------------------ teardown ------------------------------
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // a wait ran out: give copies and MMAs still in flight time to land before the memory is released
        if (tid == 0) atomicAdd(p.status + 1, 1);
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000ll) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 0) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// One plane as the loads see it (64 columns x the heads of two query rows) and as the stores do (a warp's 32 columns of one).
bool plane_maps(CUtensorMap* load, CUtensorMap* store, const void* plane, int B, int NH, int out_heads, int64_t rows, int64_t cols) {
    const uint64_t bh = (uint64_t)B * NH, ncb = (uint64_t)cols / 64, nrb = (uint64_t)rows / UNIT;
    const uint64_t dims[5] = {64, bh, (uint64_t)UNIT, ncb, nrb};
    const uint64_t str[4] = {128, bh * 128, UNIT * bh * 128, ncb * UNIT * bh * 128};
    const uint32_t in[5] = {64, (uint32_t)NH, 2, 1, 1}, out[5] = {32, (uint32_t)out_heads, 1, 1, 1};
    return make_tensor_map_bf16(load, plane, 5, dims, str, in, true) && make_tensor_map_bf16(store, plane, 5, dims, str, out, true, 64);
}

template <int NH, bool CONCAT, int BUFS>
cudaError_t launch_shape(LinkParams p, int act, const TcAlignLinkArgs& a, int64_t d_rows, int64_t d_cols, cudaStream_t stream) {
    using S = Shape<NH, CONCAT, BUFS>;
    constexpr int kSmem = 232448;   // one CTA's shared memory
    CUtensorMap maps[4];
    if (!plane_maps(maps, maps + 2, a.plane_x, a.B, NH, S::BOX, a.plane_rows, a.plane_cols)) return cudaErrorInvalidValue;
    maps[1] = maps[0]; maps[3] = maps[2];
    if (a.plane_d && !plane_maps(maps + 1, maps + 3, a.plane_d, a.B, NH, S::BOX, d_rows, d_cols)) return cudaErrorInvalidValue;
    p.stages = kMaxStages;
    while (p.stages > 2 && S::total(p.stages, p.has_d != 0, p.hid) > kSmem) --p.stages;
    const size_t smem = std::max(S::total(p.stages, p.has_d != 0, p.hid), kSmem / 2 + 1);   // one CTA per SM: it takes all of the tensor memory
    if (smem > kSmem) return cudaErrorInvalidValue;
    auto kernel = act == LISA_ACT_RELU   ? tc_align_link_kernel<NH, CONCAT, LISA_ACT_RELU, BUFS>
                  : act == LISA_ACT_SILU ? tc_align_link_kernel<NH, CONCAT, LISA_ACT_SILU, BUFS>
                                         : tc_align_link_kernel<NH, CONCAT, LISA_ACT_NONE, BUFS>;
    cudaError_t e = allow_smem(kernel, smem, true);
    if (e != cudaSuccess) return e;
    // two tiles per CTA at least: half of a CTA's time on a single tile would be the weights
    const unsigned grid = (unsigned)std::min<int64_t>((p.total + 1) / 2, sm_count());
    return launch_kernel(a.chained, kernel, dim3(grid), dim3(S::THREADS), smem, stream, p, maps[0], maps[1], maps[2], maps[3]);
}

bool link_ok(int Hq, const lisa_link& l) {
    if (l.integrate == LISA_INTEGRATE_PLUS) return Hq == 32 || Hq == 40;
    if (l.integrate == LISA_INTEGRATE_CONCAT) {
        if (Hq != 32) return false;
        return l.ffn_layers == 2 ? (l.m >= 1 && l.m <= 256) : l.m == Hq;
    }
    if (Hq != 32 && Hq != 40) return false;
    return l.ffn_layers == 2 ? (l.m >= 1 && l.m <= 256) : l.m == Hq;
}

}  // namespace

bool tc_align_concat_supported(int Hq, const lisa_link* links, int chain) {
    if (chain < 1) return false;
    for (int k = 0; k < chain; ++k)
        if (links[k].integrate != LISA_INTEGRATE_CONCAT || !link_ok(Hq, links[k])) return false;
    return true;
}

// Chains of adding (or FFN-free) links, one launch per link: 32 or 40 heads, hidden width up to 256.
bool tc_align_link_supported(int Hq, const lisa_link* links, int chain) {
    if (chain < 1) return false;
    for (int k = 0; k < chain; ++k)
        if (links[k].integrate == LISA_INTEGRATE_CONCAT || !link_ok(Hq, links[k])) return false;
    return true;
}

cudaError_t launch_tc_align_link(const TcAlignLinkArgs& a, cudaStream_t stream) {
    if (a.plane_cols % 64 != 0 || a.plane_rows % 128 != 0) return cudaErrorInvalidValue;
    const lisa_link& l = *a.link;
    if (!link_ok(a.Hq, l)) return cudaErrorInvalidValue;
    const bool concat = l.integrate == LISA_INTEGRATE_CONCAT;
    if (concat && !a.plane_d) return cudaErrorInvalidValue;
    LinkParams p{};
    p.N = a.N; p.row0 = a.row0 >= 0 ? a.row0 : a.qt_begin * UNIT;
    if (p.row0 % UNIT != 0 || p.row0 > a.qt_begin * UNIT) return cudaErrorInvalidValue;
    const int64_t d_cols = a.d_plane_cols > 0 ? a.d_plane_cols : a.plane_cols;
    p.d_row0 = a.d_plane_cols > 0 ? (a.d_row0 >= 0 ? a.d_row0 : a.qt_begin * UNIT) : p.row0;
    if (d_cols % 64 != 0 || p.d_row0 % UNIT != 0 || p.d_row0 > a.qt_begin * UNIT || (a.d_plane_cols > 0 && a.d_plane_rows % 128 != 0))
        return cudaErrorInvalidValue;
    p.row_begin = a.qt_begin * UNIT;
    p.row_end = std::min(a.N, (a.qt_begin + a.qt_count) * UNIT);
    if (p.row_end <= p.row_begin) return cudaErrorInvalidValue;
    int64_t tiles = 0;
    for (int r = p.row_begin; r < p.row_end; r += 64) tiles += (int64_t)((std::min(p.row_end - r, 64) + 1) / 2) * (r / 64 + 1);
    if (tiles * a.B > 0x3fffffff) return cudaErrorInvalidValue;
    p.tiles_per_batch = (int)tiles;
    p.total = (int)tiles * a.B;
    p.has_d = a.plane_d != nullptr;
    const int64_t d_rows = a.d_plane_cols > 0 ? a.d_plane_rows : a.plane_rows;
    p.status = status_words();
    if (!p.status) return cudaErrorUnknown;
    p.dst_next = a.dst_next; p.dst_scaled = a.dst_scaled;
    p.w1 = l.w1; p.b1 = l.b1; p.w2 = l.w2; p.b2 = l.b2; p.w_dtype = l.w_dtype;
    p.kind = alignmma::link_kind(l.integrate, l.ffn_layers);
    p.m = l.m;
    const int act = p.kind == KIND_FFN ? l.act : LISA_ACT_NONE;
    const int inputs = concat ? 2 * a.Hq : a.Hq;
    p.hid = ((p.kind == KIND_FFN ? l.m : inputs) + 15) / 16 * 16;
    // Four tiles in flight as long as a quarter of the tensor memory holds a tile's hidden layer (128 units), two above.
    cudaError_t e;
    if (concat) e = p.hid <= 128 ? launch_shape<32, true, 4>(p, act, a, d_rows, d_cols, stream) : launch_shape<32, true, 2>(p, act, a, d_rows, d_cols, stream);
    else if (a.Hq == 32) e = p.hid <= 128 ? launch_shape<32, false, 4>(p, act, a, d_rows, d_cols, stream) : launch_shape<32, false, 2>(p, act, a, d_rows, d_cols, stream);
    else e = p.hid <= 128 ? launch_shape<40, false, 4>(p, act, a, d_rows, d_cols, stream) : launch_shape<40, false, 2>(p, act, a, d_rows, d_cols, stream);
    count_launches(1);
    return e;
}

}  // namespace lisa
