// Tensor-core flash kernel (tcgen05 + TMEM + TMA) for head width 128, bf16.
//
// One CTA per (batch b, query head h, 128-row query tile).  For every 64-key tile j up to the diagonal:
//   scores  S = QA . KA^T            tcgen05.mma (M 128, N 64), fp32 accumulator in tensor memory, two buffers
//   logits  A = S * scale (+ Y)      Y: optional fp16 tile of pre-computed scores (the aligned part of a
//                                    shared layer, Eq. 4; then QA/KA are the layer's low-rank Q'/K', Eq. 3)
//   causal mask (tiles that reach past the first query row), online softmax in registers (one thread per query
//   row), P as bf16
//   O += P . V                       tcgen05.mma (M 128, N 128, K 64), V read MN-major straight from its [key][d] tile
// With QA/KA = Q/K and no Y this is standard attention (Eq. 1-2).  In MODE_EMIT there is no softmax: the scaled
// scores leave as fp16 tiles (staged in shared memory, stored with TMA) for the aligner kernel.  In MODE_ATTN_CARRY the
// attention also writes its finished pre-softmax logits A = S * scale + Y (unmasked, Eq. 4's A_n) back as fp16 tiles: the
// next shared layer of a chain aligns those instead of recomputing the chain from the anchor's scores.
//
// Warp roles: warps 0-3 and 4-7 softmax/epilogue (thread = query row = TMEM lane; the two warpgroups take the key tiles in turn), warp 8
// TMA producer, warp 9 issuer of the score MMAs and TMEM owner, warp 10 issuer of the P.V MMAs (warp 11 only completes the warpgroup).
// A K stage is free again as soon as its score MMA has run, a Y stage once its rows are read, a V stage after the P.V MMA; where P lies, see
// Smem::P_SMEM.
// Sizing: a softmax warp spends as long on waits (tensor memory, barriers, the next scores behind P.V) as on its 64 exponentials a row (16
// lanes a cycle and SM: 512 cycles a tile), so an SM partition needs four of them in different phases: TWO CTAs share an SM (64-key tiles
// keep a CTA at 112 KB of shared memory and 256 tensor-memory columns), each with two warpgroups on alternate tiles.  One warpgroup
// per CTA took 1010 cycles a tile and SM, two warpgroups on halves of the same tile as long (in step, they wait for the same unit at the
// same time), alternate tiles 845.  A row's reference maximum is handed on behind the exponentials, which keeps the two warpgroups of a CTA
// from coming to theirs together.  Attention with plane, 2048 tokens of 32 heads 53.6 -> 51.6 us captured cold (of which 3 are the first loads of
// 296 CTAs at a time, 22 MB, and 8 the tail); 2 x 1777 of 40 heads, with and without write-back 241 -> 228; 4 x 8192 3.6 -> 3.1 ms without.
// Every wait is bounded; on expiry the CTA records it in the status word, drains and exits.
#include "common.cuh"
#include "tc_common.cuh"

namespace lisa {
namespace {

using namespace tc;

constexpr int BM = 128, BN = 64, D = 128;

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

constexpr int kPrefetchAhead = 2;   // tiles (0: no L2 prefetch)
constexpr int kSoftmaxWarps = 8;
constexpr int kThreads = 384;   // warpgroups 0 and 1: softmax/epilogue; warpgroup 2: producer, two MMA issuers, one idle warp

struct FlashParams {
    int B, N, Hq, Hkv;
    float scale_log2;  // score scale * log2(e)
    __nv_bfloat16* o;
    int64_t o_sb, o_sn, o_sh;
    int* status;
    int plane_row0;  // first query row held by the plane workspace (rows are stored relative to it)
    int qt_begin;    // this launch covers query tiles [qt_begin, qt_begin + gridDim.y)
    int ksteps;      // 16-wide k-steps of the score MMA actually issued (<= KD/16; the rest is zero padding)
    float scale;     // MODE_EMIT: scores are multiplied by this before rounding to fp16
};

// MODE_ATTN: softmax(QA.KA^T).V;  MODE_ATTN_PLANE: the same with the pre-computed tile Y added to the logits
// (Y arrives already multiplied by log2(e));  MODE_EMIT: no softmax, the scaled scores go to the plane workspace;
// MODE_ATTN_CARRY: MODE_ATTN_PLANE that also stores the logits (divided by log2(e) again) through the fifth tensor map.
constexpr int MODE_ATTN = 0, MODE_ATTN_PLANE = 1, MODE_EMIT = 2, MODE_ATTN_CARRY = 3;

template <int KD, int MODE>
struct Smem {
    static constexpr bool PLANE = MODE == MODE_ATTN_PLANE || MODE == MODE_ATTN_CARRY;
    static constexpr bool EMIT = MODE == MODE_EMIT;
    static constexpr bool CARRY = MODE == MODE_ATTN_CARRY;
    // Where P lies: over the scores it came from, in tensor memory, as a tensor-memory operand of P.V, or in shared memory.  Over the scores,
    // S(t + 2) has to wait for P(t).V(t), 1300 of a warpgroup's 3700 cycles a tile; in shared memory it need not, but there is room for that
    // only beside a plane that is not written back (a written one has its logits over Y until the copy engine has read them: four stages).
    static constexpr bool P_SMEM = MODE == MODE_ATTN_PLANE;
    static constexpr int KST = EMIT || KD == 128 ? 3 : 2;  // K ring depth
    static constexpr int VST = 2;                  // V ring depth
    static constexpr int RB = KD == 128 ? 128 : 64;   // bytes of a row of a Q or K tile: 64 of the 128 columns, or all 32
    static constexpr int YST = !PLANE ? 0 : P_SMEM ? 2 : 4;   // Y ring depth
    static constexpr int Q_BYTES = BM * KD * 2;
    static constexpr int K_BYTES = BN * KD * 2;
    static constexpr int V_BYTES = EMIT ? 0 : BN * D * 2;
    static constexpr int Y_BYTES = PLANE ? BM * BN * 2 : 0;
    static constexpr int STG_BYTES = EMIT ? kSoftmaxWarps * 4096 : 0;   // emit: [32 rows][128 B] per epilogue warp
    static constexpr int OFF_Q = 0;
    static constexpr int OFF_K = OFF_Q + Q_BYTES;
    static constexpr int OFF_V = OFF_K + KST * K_BYTES;
    static constexpr int OFF_Y = OFF_V + VST * V_BYTES;
    static constexpr int P_BYTES = P_SMEM ? BM * BN * 2 : 0;
    static constexpr int OFF_P = OFF_Y + YST * Y_BYTES;
    static constexpr int OFF_STG = OFF_P + 2 * P_BYTES;
    static constexpr int OFF_M = OFF_STG + STG_BYTES;      // reference maximum of each row: [128] fp32
    static constexpr int OFF_BAR = OFF_M + (EMIT ? 0 : BM * 4);
    static constexpr int TOTAL = OFF_BAR + 320;
    static constexpr uint32_t TMEM_COLS = EMIT ? 128 : 256;   // S[2]: [0,128), O: [128,256)
    static_assert(TOTAL <= 115712, "two CTAs must fit one SM's shared memory");
};

template <int KD, int MODE>
__global__ void __launch_bounds__(kThreads, 2)
tc_flash_kernel(const __grid_constant__ FlashParams p, const __grid_constant__ CUtensorMap tmQ,
                const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmC) {
    using L = Smem<KD, MODE>;
    constexpr bool PLANE = L::PLANE, EMIT = L::EMIT, CARRY = L::CARRY;
    constexpr int KST = L::KST;
    extern __shared__ __align__(1024) uint8_t smem[];
    // 128-byte-swizzled tiles need 1024-byte aligned bases; the dynamic window starts on such a boundary (there is no
    // static shared memory in this kernel).  Should that ever not hold, refuse loudly instead of computing garbage.
    if ((smem_u32(smem) & 1023u) != 0) {
        if (threadIdx.x == 0) atomicAdd(p.status + 1, 1);
        return;
    }
    uint8_t* sQ = smem + L::OFF_Q;
    uint8_t* sK = smem + L::OFF_K;
    uint8_t* sV = smem + L::OFF_V;
    uint8_t* sY = smem + L::OFF_Y;
    uint8_t* sP = smem + L::OFF_P;
    uint8_t* sStg = smem + L::OFF_STG;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::OFF_BAR);
    uint64_t* q_full = bars + 0;
    uint64_t* k_full = bars + 1;    // [KST <= 3]
    uint64_t* k_empty = bars + 4;   // [KST <= 3]
    uint64_t* v_full = bars + 7;    // [VST <= 2]
    uint64_t* y_full = bars + 9;    // [YST <= 4]
    uint64_t* y_empty = bars + 13;  // [YST <= 4] Y rows read (carry: and the logits that went over them stored)
    uint64_t* s_full = bars + 17;   // [2] score buffer written by the MMA
    uint64_t* s_free = bars + 19;   // [2] emit, P_SMEM: score buffer copied to registers (else free with pv_done)
    uint64_t* p_full = bars + 21;   // [2] P is there
    uint64_t* pv_done = bars + 23;  // [2] P.V has run: the place of P is free
    uint64_t* m_set = bars + 25;    // [2][4] the rows of a quarter have their reference maximum for a tile
    uint64_t* v_empty = bars + 33;  // [VST] P.V of the tile in the stage has run
    uint64_t* o_full = bars + 35;   // the last P.V has run (a barrier of its own: pv_done tells only neighbouring phases apart)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 36);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 37);

    const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
    // blockIdx.x (the fastest-dispatched index) runs over a group of (batch, head) pairs, blockIdx.y over query tiles from the last one
    // down: every CTA of a group's heaviest tile is handed out before any lighter one, so the SMs finish close together.  blockIdx.z runs
    // over the groups: see launch_tc_flash.
    const int qt = p.qt_begin + (int)gridDim.y - 1 - (int)blockIdx.y;
    const int bh = (int)(blockIdx.z * gridDim.x + blockIdx.x);
    const int h = bh % p.Hq, b = bh / p.Hq;
    const int g = h / (p.Hq / p.Hkv);
    const int q0 = qt * BM;
    const int nt = min((q0 + BM) / BN, (p.N + BN - 1) / BN);  // key tiles 0..nt-1 reach the last query row / the last key

    constexpr int NQ = KD * 2 / L::RB, NK = NQ, NV = EMIT ? 0 : D / 64;   // copies of a tile
    auto load_k = [&](int t, int stage) {
        mbar_expect_tx(k_full + stage, L::K_BYTES);
#pragma unroll
        for (int i = 0; i < NK; ++i) tma_load_4d(sK + stage * L::K_BYTES + i * (BN * L::RB), &tmK, k_full + stage, i * 64, g, t * BN, b);
    };
    auto load_y = [&](int t, int stage) {
        mbar_expect_tx(y_full + stage, L::Y_BYTES);
        tma_load_5d(sY + stage * L::Y_BYTES, &tmY, y_full + stage, 0, b * p.Hq + h, 0, t, (q0 - p.plane_row0) / BM);
    };
    if (warp == kSoftmaxWarps + 1) tmem_alloc(tmem_slot, L::TMEM_COLS);
    if (warp == kSoftmaxWarps) {   // a barrier to a lane: q, k, v, y full and empty, s, p and pv, m, v empty, o in the order of `bars`
        auto count = [](int i) {
            const bool four = (i >= 13 && i < 17) || (i >= 19 && i < 23);   // y_empty; s_free and p_full: the warps of a warpgroup
            return four ? 4 : 1;
        };
        mbar_init(bars + lane, count(lane));
        if (lane < 4) mbar_init(bars + 32 + lane, count(32 + lane));
        if (lane == 0) *abort_flag = 0;
        fence_barrier_init();
        if (elect_one()) {
            tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK);
            if (!EMIT) tma_prefetch_desc(&tmV);
            if (PLANE || EMIT) tma_prefetch_desc(&tmY);
            if (CARRY) tma_prefetch_desc(&tmC);
        }
        __syncwarp();
    }
    // What comes before -- barriers, tensor memory, the tensor maps (arguments of the launch) -- overlaps the tail of the kernel before this one.
    chain_wait();
    // The first tiles are on their way before the CTA has come together (barriers a lane each, in the loader's warp): a CTA's first scores wait for
    // nothing else.  A CTA of 2048 tokens spends a third of its time outside its loop over tiles; 197 tokens through an anchor and three
    // layers 74.7 -> 73.5 us, an anchor and three layers of 4 x 8192 1.5 % less.
    if (warp == kSoftmaxWarps) {
        if (elect_one()) {
            mbar_expect_tx(q_full, L::Q_BYTES);
#pragma unroll
            for (int i = 0; i < NQ; ++i) tma_load_4d(sQ + i * (BM * L::RB), &tmQ, q_full, i * 64, h, q0, b);
            load_k(0, 0);
            if constexpr (PLANE) load_y(0, 0);
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    chain_release();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const uint32_t tmem_O = tmem_base + 128;

    // The kernel is compiled for 80 registers per thread (two CTAs of 384 threads per SM).  A softmax thread holds 64 scores; the
    // single-thread roles need few: warpgroup 2 hands registers back and the softmax warpgroups take them (256 x 104 + 128 x 32 = 384 x 80).
    if (warp >= kSoftmaxWarps) {
    if constexpr (!EMIT) asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (warp == kSoftmaxWarps) {
        // ------------------------------ TMA producer ------------------------------
        // Round t brings K(t) and Y(t), then V(t - 1): V is needed a softmax pass later than the others, and asked for in its own round
        // its stage, which waits for the P.V two tiles before, would hold up the Y of the next.
        int ks = 0, ys = 0, vs = 0;      // K and Y stage of tile t, V stage of tile t - 1
        uint32_t kpar = 1, ypar = 1, vpar = 1;     // parity to wait for on their "empty" barriers (first pass: passes at once)
        for (int t = 0; t < nt + (EMIT ? 0 : 1); ++t) {
            bool okp = true;
            if (t > 0 && t < nt) {   // (the first tile has been asked for above)
                okp = mbar_wait(k_empty + ks, kpar, abort_flag);
                if (!__all_sync(0xffffffffu, okp)) break;
                if (elect_one()) load_k(t, ks);
                __syncwarp();
                if constexpr (PLANE) {
                    okp = mbar_wait(y_empty + ys, ypar, abort_flag);
                    if (!__all_sync(0xffffffffu, okp)) break;
                    if (elect_one()) load_y(t, ys);
                    __syncwarp();
                }
            }
            if constexpr (!EMIT) {
                if (t > 0) {
                    okp = mbar_wait(v_empty + vs, vpar, abort_flag);
                    if (!__all_sync(0xffffffffu, okp)) break;
                    if (elect_one()) {
                        mbar_expect_tx(v_full + vs, L::V_BYTES);
#pragma unroll
                        for (int i = 0; i < NV; ++i) tma_load_4d(sV + vs * L::V_BYTES + i * (BN * 128), &tmV, v_full + vs, i * 64, g, (t - 1) * BN, b);
                    }
                    __syncwarp();
                    if (++vs == L::VST) { vs = 0; vpar ^= 1; }
                }
            }
            // The V and Y stages can be refilled at most two softmax passes before they are needed, under load less than a trip to HBM.
            // Their tiles are therefore asked into L2 earlier, kPrefetchAhead tiles ahead of the one just issued.
            if constexpr (kPrefetchAhead > 0 && !EMIT) {
                if (t + kPrefetchAhead < nt && elect_one()) {
#pragma unroll
                    for (int i = 0; i < NV; ++i) tma_prefetch_l2_4d(&tmV, i * 64, g, (t + kPrefetchAhead) * BN, b);
                    if constexpr (PLANE) tma_prefetch_l2_5d(&tmY, 0, b * p.Hq + h, 0, t + kPrefetchAhead, (q0 - p.plane_row0) / BM);
                }
                __syncwarp();
            }
            if (++ks == KST) { ks = 0; kpar ^= 1; }
            if (PLANE && ++ys == L::YST) { ys = 0; ypar ^= 1; }
        }
    } else if (warp == kSoftmaxWarps + 1) {
        // ------------------------------ MMA issuer: scores ------------------------------
        // Issuing a tcgen05.mma holds the issuing thread for about as long as the MMAs queued before it take to run, so
        // the score MMAs and the P.V MMAs are issued by two different warps: each waits for its own operands and the
        // two hold-ups overlap instead of adding up.  Every lane of an issuing warp runs the loop (waits, stage
        // counters, descriptor arithmetic: all warp-uniform); only the MMA and commit instructions themselves are
        // issued by one elected lane.
        constexpr uint32_t IDESC_QK = umma_idesc_bf16(BM, BN, 0, 0);
        const int ksteps = p.ksteps;
        // Descriptors are built once; per MMA only the start-address field (bits 0-13 of the low word, in
        // 16-byte units) moves, by a compile-time constant or a stage offset: no carry can leave the field.
        auto desc_off = [](uint64_t d, uint32_t bytes) -> uint64_t {
            return (d & 0xffffffff00000000ull) | (uint32_t)((uint32_t)d + (bytes >> 4));
        };
        const uint64_t dq0 = KD == 128 ? umma_desc_sw128(smem_u32(sQ), 16, 1024) : umma_desc_sw64(smem_u32(sQ));
        const uint64_t dk0 = KD == 128 ? umma_desc_sw128(smem_u32(sK), 16, 1024) : umma_desc_sw64(smem_u32(sK));
        // scores of tile t into buffer t&1; needs K(t) loaded and (t >= 2) the buffer: the scores of t-2 read, or P(t-2), which lies there,
        // multiplied
        uint64_t* buf_free = EMIT || L::P_SMEM ? s_free : pv_done;
        int sk = 0;
        uint32_t kpar = 0;
        bool ok = __all_sync(0xffffffffu, mbar_wait(q_full, 0, abort_flag));
        for (int t = 0; ok && t < nt; ++t) {
            const int s = t & 1;
            ok = mbar_wait(k_full + sk, kpar, abort_flag) && mbar_wait(buf_free + s, ((t >> 1) & 1) ^ 1, abort_flag);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;   // one verdict for the whole warp
            tc_fence_after();
            const uint64_t dk = desc_off(dk0, sk * L::K_BYTES);
            const uint32_t dst = tmem_base + s * BN;
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < KD / 16; ++ks) {
                    if (ks < ksteps)
                        umma_ss(dst, desc_off(dq0, (ks >> 2) * (BM * L::RB) + (ks & 3) * 32), desc_off(dk, (ks >> 2) * (BN * L::RB) + (ks & 3) * 32), IDESC_QK, ks > 0);
                }
                umma_commit(s_full + s);
                if (t + KST < nt) umma_commit(k_empty + sk);  // nobody waits for the last ones: do not arm them
            }
            __syncwarp();
            if (++sk == KST) { sk = 0; kpar ^= 1; }
        }
    } else if (warp == kSoftmaxWarps + 2) {
        // ------------------------------ MMA issuer: P.V ------------------------------
        if constexpr (!EMIT) {
            constexpr uint32_t IDESC_PV = umma_idesc_bf16(BM, D, 0, 1);
            auto desc_off = [](uint64_t d, uint32_t bytes) -> uint64_t {
                return (d & 0xffffffff00000000ull) | (uint32_t)((uint32_t)d + (bytes >> 4));
            };
            const uint64_t dv0 = umma_desc_sw128(smem_u32(sV), BN * 128, 1024);
            const uint64_t dp0 = umma_desc_sw128(smem_u32(sP), 16, 1024);
            bool ok = true;
            int vs = 0;
            uint32_t vpar = 0;
            for (int t = 0; ok && t < nt; ++t) {
                const int s = t & 1;
                ok = mbar_wait(v_full + vs, vpar, abort_flag) && mbar_wait(p_full + s, (t >> 1) & 1, abort_flag);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                tc_fence_after();
                const uint64_t dv = desc_off(dv0, vs * L::V_BYTES);
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < BN / 16; ++ks) {
                        // P: two keys a column, or K-major, 64 keys per 128-byte row; V: 16 keys = two 8-row groups, the next 64 d-columns BN * 128 bytes further on
                        if constexpr (L::P_SMEM) umma_ss(tmem_O, desc_off(dp0, s * L::P_BYTES + ks * 32), desc_off(dv, ks * 2048), IDESC_PV, (t > 0) || (ks > 0));
                        else umma_ts(tmem_O, tmem_base + s * BN + ks * 8, desc_off(dv, ks * 2048), IDESC_PV, (t > 0) || (ks > 0));
                    }
                    umma_commit(pv_done + s);
                    if (t + L::VST < nt) umma_commit(v_empty + vs);
                    if (t + 1 == nt) umma_commit(o_full);
                }
                __syncwarp();
                if (++vs == L::VST) { vs = 0; vpar ^= 1; }
            }
        }
    }
    } else if constexpr (EMIT) {
        // ------------------------------ epilogue: warps 0-3 even tiles, 4-7 odd ones (thread = query row) ------------------------------
        const int q = warp & 3, s = warp >> 2;
        const uint32_t lane_sel = (uint32_t)(q * 32) << 16;
        const float emit_scale = p.scale;
        uint8_t* stg = sStg + warp * 4096;
        for (int t = s; t < nt; t += 2) {
            if (!__all_sync(0xffffffffu, mbar_wait(s_full + s, (t >> 1) & 1, abort_flag))) break;
            tc_fence_after();
            uint32_t sr[BN];
#pragma unroll
            for (int c = 0; c < BN / 32; ++c) tmem_ld32(tmem_base + s * BN + lane_sel + c * 32, sr + c * 32);
            tmem_wait_ld();
            tc_fence_before();
            if (lane == 0) tma_store_wait_read<0>();  // the store of tile t-2 has read this buffer
            __syncwarp();
            if (lane == 0) mbar_arrive(s_free + s);
            const float2* sf = reinterpret_cast<const float2*>(sr);
            // this warp's 32 rows x 64 columns as fp16 into its staging buffer (swizzled like any other tile), then lane 0 stores it
#pragma unroll
            for (int c = 0; c < BN / 8; ++c) {
                uint32_t v[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 x = __fmul2_rn(sf[c * 4 + e], make_float2(emit_scale, emit_scale));
                    v[e] = pack_f16(x.x, x.y);
                }
                *reinterpret_cast<uint4*>(stg + sw128_offset(lane, c)) = make_uint4(v[0], v[1], v[2], v[3]);
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                tma_store_5d(&tmY, stg, 0, b * p.Hq + h, q * 32, t, (q0 - p.plane_row0) / BM);
                tma_store_commit();
            }
        }
        if (lane == 0) tma_store_wait_all<0>();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
        // ------------------------------ softmax / epilogue (thread = query row = TMEM lane) ------------------------------
        // The two warpgroups take the key tiles in turn, so that the four softmax warps of an SM partition (two CTAs) are in different
        // phases: one waits for tensor memory or for its next scores while another keeps the transcendental unit busy.
        const int q = warp & 3, wg = warp >> 2;
        const int row = q * 32 + lane;             // 0..127
        const int qi = q0 + row;                   // global query index
        const uint32_t lane_sel = (uint32_t)(q * 32) << 16;
        const float scale_log2 = p.scale_log2;
        volatile float* m_row = reinterpret_cast<float*>(smem + L::OFF_M) + row;
        float m_ref = -INFINITY, l_sum = 0.f;
        bool ok = true;
        int ys = wg;                               // Y stage and the parity of its barrier
        uint32_t ypar = 0;
        for (int t = wg; t < nt; t += 2) {
            const int s = wg;
            if (!(ok = __all_sync(0xffffffffu, mbar_wait(s_full + s, (t >> 1) & 1, abort_flag)))) break;
            tc_fence_after();
            uint32_t sr[BN];
#pragma unroll
            for (int c = 0; c < BN / 32; ++c) tmem_ld32(tmem_base + s * BN + lane_sel + c * 32, sr + c * 32);
            float* sf = reinterpret_cast<float*>(sr);
            if constexpr (PLANE) {
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(y_full + ys, ypar, abort_flag)))) break;
                uint8_t* yb = sY + ys * L::Y_BYTES;
                tmem_wait_ld();
                if constexpr (L::P_SMEM) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(s_free + s);
                }
#pragma unroll
                for (int c = 0; c < BN / 8; ++c) {
                    const uint4 y = *reinterpret_cast<const uint4*>(yb + sw128_offset(row, c));
                    const uint32_t w[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float2* s2 = reinterpret_cast<float2*>(sf) + c * 4 + e;
                        *s2 = __ffma2_rn(*s2, make_float2(scale_log2, scale_log2), unpack_f16(w[e]));
                    }
                    if constexpr (CARRY) {
                        // the finished logits go over the row's Y as fp16 (back in the natural-log domain, before the mask: the next
                        // layer's aligner sees finite values everywhere) and from there to the scores buffer
                        constexpr float kLn2 = 0.6931471805599453f;
                        uint32_t v[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 x = __fmul2_rn(reinterpret_cast<const float2*>(sf)[c * 4 + e], make_float2(kLn2, kLn2));
                            v[e] = pack_f16(x.x, x.y);
                        }
                        *reinterpret_cast<uint4*>(yb + sw128_offset(row, c)) = make_uint4(v[0], v[1], v[2], v[3]);
                    }
                }
                if constexpr (CARRY) fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if constexpr (CARRY) {
                        tma_store_5d(&tmC, yb + q * 4096, 0, b * p.Hq + h, q * 32, t, (q0 - p.plane_row0) / BM);
                        tma_store_commit();
                    } else {
                        mbar_arrive(y_empty + ys);
                    }
                }
            } else {
                tmem_wait_ld();
            }
            // from here on: PLANE -> sf holds log2-domain logits; otherwise raw scores, scaled inside the exp
            if (t * BN + BN - 1 > q0) {   // the tile reaches past the CTA's first query row: mask keys after each row
#pragma unroll
                for (int j = 0; j < BN; ++j)
                    if (t * BN + j > qi) sf[j] = -INFINITY;
            }
            float mx[4] = {sf[0], sf[1], sf[2], sf[3]};   // four independent chains instead of one of 64 dependent steps
#pragma unroll
            for (int j = 4; j + 8 <= BN; j += 8) {   // two new values per step and chain: a three-input maximum where there is one
                mx[0] = fmaxf(fmaxf(mx[0], sf[j]), sf[j + 4]); mx[1] = fmaxf(fmaxf(mx[1], sf[j + 1]), sf[j + 5]);
                mx[2] = fmaxf(fmaxf(mx[2], sf[j + 2]), sf[j + 6]); mx[3] = fmaxf(fmaxf(mx[3], sf[j + 3]), sf[j + 7]);
            }
            mx[0] = fmaxf(mx[0], sf[BN - 4]); mx[1] = fmaxf(mx[1], sf[BN - 3]);
            mx[2] = fmaxf(mx[2], sf[BN - 2]); mx[3] = fmaxf(mx[3], sf[BN - 1]);
            float m_t = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
            if constexpr (!PLANE) m_t *= scale_log2;
            // The reference maximum of a row goes from tile to tile, that is from one warpgroup to the other, through shared memory.  Lazy
            // rescale: it moves only when some row of the warp outgrew it by 2^8 (a row with every key of this tile masked has m_t = -inf
            // and never asks for it); then the accumulator is rescaled, after every P.V issued so far has landed in it.
            float m_new = -INFINITY;
            if (t > 0) {
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(m_set + (wg ^ 1) * 4 + q, ((t - 1) >> 1) & 1, abort_flag)))) break;
                m_new = *m_row;
            }
            const float m_old = m_new;
            const bool rescale = __any_sync(0xffffffffu, m_t > m_new + 8.f) || t == 0;
            if (rescale) {
                m_new = fmaxf(m_new, m_t);
                *m_row = m_new;
            }
            // P(t - 2) has been multiplied: its place is free, and p_full, whose phases the P.V warp tells apart by parity alone, cannot run ahead
            if (L::P_SMEM && t >= 2 && !(ok = __all_sync(0xffffffffu, mbar_wait(pv_done + s, ((t - 2) >> 1) & 1, abort_flag)))) break;
            const float mine = fast_exp2(m_ref - m_new);   // this warpgroup's sum so far: 1 unless the reference has moved since
            m_ref = m_new;
            if (t > 0 && rescale) {
                const float factor = fast_exp2(m_old - m_new);
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(pv_done + (wg ^ 1), ((t - 1) >> 1) & 1, abort_flag)))) break;
                tc_fence_after();
#pragma unroll 1
                for (int c = 0; c < D / 16; ++c) {
                    uint32_t orr[16];
                    tmem_ld16(tmem_O + lane_sel + c * 16, orr);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float2* o2 = reinterpret_cast<float2*>(orr) + j;
                        *o2 = __fmul2_rn(*o2, make_float2(factor, factor));
                    }
                    tmem_st16(tmem_O + lane_sel + c * 16, orr);
                }
            }
            // The fp32 arithmetic around the exponentials runs two values per instruction (packed fp32 pairs; the scores of a thread sit in
            // consecutive registers).
            float2 sum2 = make_float2(0.f, 0.f);
            const float2 neg_m2 = make_float2(-m_ref, -m_ref), scale2 = make_float2(scale_log2, scale_log2);
            const float2* sf2 = reinterpret_cast<const float2*>(sf);
#pragma unroll
            for (int c = 0; c < BN / 32; ++c) {
                uint32_t pk[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float2 x = PLANE ? __fadd2_rn(sf2[c * 16 + j], neg_m2) : __ffma2_rn(sf2[c * 16 + j], scale2, neg_m2);
                    const float2 e = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                    sum2 = __fadd2_rn(sum2, e);
                    pk[j] = pack_bf16(e.x, e.y);
                }
                if constexpr (L::P_SMEM) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        *reinterpret_cast<uint4*>(sP + s * L::P_BYTES + sw128_offset(row, c * 4 + j)) = make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
                } else {
                    tmem_st16(tmem_base + s * BN + lane_sel + c * 16, pk);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(m_set + wg * 4 + q);
            l_sum = l_sum * mine + (sum2.x + sum2.y);
            tmem_wait_st();   // (P, or a rescaled accumulator)
            tc_fence_before();
            if constexpr (L::P_SMEM) fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(p_full + s);
                if constexpr (CARRY) {
                    tma_store_wait_read<0>();   // the logits have left: the stage may be refilled
                    mbar_arrive(y_empty + ys);
                }
            }
            if (PLANE) {
                if ((ys += 2) >= L::YST) { ys -= L::YST; ypar ^= 1; }
            }
        }
        if constexpr (CARRY) {
            if (lane == 0) tma_store_wait_all<0>();
        }
        // The row's sum: both warpgroups' shares on the last reference maximum, through the Q tile, which nobody reads any more once
        // the last P.V has run.  Every softmax warp comes to the barrier, one whose wait ran out as well.
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(o_full, 0, abort_flag));
        float* l_x = reinterpret_cast<float*>(sQ);
        if (ok) l_x[wg * BM + row] = l_sum * fast_exp2(m_ref - *m_row);
        asm volatile("barrier.cta.sync 1, 256;" ::: "memory");
        if (ok) {
            tc_fence_after();
            const float inv_l = 1.f / (l_x[row] + l_x[BM + row]);
            __nv_bfloat16* orow = p.o + b * p.o_sb + (int64_t)qi * p.o_sn + h * p.o_sh + wg * (D / 2);
#pragma unroll
            for (int c = 0; c < D / 2 / 32; ++c) {
                uint32_t orr[32];
                tmem_ld32(tmem_O + lane_sel + wg * (D / 2) + c * 32, orr);
                tmem_wait_ld();
                if (qi < p.N) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint4 v;
                        v.x = pack_bf16(__uint_as_float(orr[k * 8 + 0]) * inv_l, __uint_as_float(orr[k * 8 + 1]) * inv_l);
                        v.y = pack_bf16(__uint_as_float(orr[k * 8 + 2]) * inv_l, __uint_as_float(orr[k * 8 + 3]) * inv_l);
                        v.z = pack_bf16(__uint_as_float(orr[k * 8 + 4]) * inv_l, __uint_as_float(orr[k * 8 + 5]) * inv_l);
                        v.w = pack_bf16(__uint_as_float(orr[k * 8 + 6]) * inv_l, __uint_as_float(orr[k * 8 + 7]) * inv_l);
                        *reinterpret_cast<uint4*>(orow + c * 32 + k * 8) = v;
                    }
                }
            }
        }
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
    if (warp == kSoftmaxWarps + 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, L::TMEM_COLS);
    }
}

}  // namespace

bool make_tensor_map_bf16(CUtensorMap* map, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes,
                          const uint32_t* box, bool fp16, int swizzle) {
    typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                 const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static EncodeFn encode = nullptr;
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
            qres != cudaDriverEntryPointSuccess)
            return false;
        encode = reinterpret_cast<EncodeFn>(fn);
    }
    cuuint64_t gdims[5], gstr[4];
    cuuint32_t gbox[5], estr[5];
    for (int i = 0; i < rank; ++i) { gdims[i] = dims[i]; gbox[i] = box[i]; estr[i] = 1; }
    for (int i = 0; i + 1 < rank; ++i) gstr[i] = strides_bytes[i];
    return encode(map, fp16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), gdims, gstr, gbox, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {
bool tma_ok(const lisa_tensor& t) {
    return t.dtype == LISA_BF16 && (reinterpret_cast<uintptr_t>(t.ptr) & 15u) == 0 && t.stride_b % 8 == 0 && t.stride_n % 8 == 0 &&
           t.stride_h % 8 == 0 && t.stride_b > 0 && t.stride_n > 0 && t.stride_h > 0;
}
// boxes of 64 columns, or of all 32
bool map_bnhx(CUtensorMap* m, const lisa_tensor& t, int B, int N, int H, int X, int rows) {
    const uint64_t dims[4] = {(uint64_t)X, (uint64_t)H, (uint64_t)N, (uint64_t)B};
    const uint64_t str[3] = {(uint64_t)t.stride_h * 2, (uint64_t)t.stride_n * 2, (uint64_t)t.stride_b * 2};
    const uint32_t box[4] = {(uint32_t)std::min(X, 64), 1, (uint32_t)rows, 1};
    return make_tensor_map_bf16(m, t.ptr, 4, dims, str, box, false, X == 32 ? 64 : 128);
}
}  // namespace

bool tc_flash_supported(const TcFlashArgs& a) {
    if (!((a.kd == 128 || a.kd == 32) && tma_ok(a.qa) && tma_ok(a.ka) && a.Hq % a.Hkv == 0)) return false;
    return a.emit_plane ? true : (tma_ok(a.v) && tma_ok(a.o));
}

cudaError_t launch_tc_flash(const TcFlashArgs& a, cudaStream_t stream) {
    CUtensorMap tmQ, tmK, tmV, tmY;
    if (!map_bnhx(&tmQ, a.qa, a.B, a.N, a.Hq, a.kd, BM) || !map_bnhx(&tmK, a.ka, a.B, a.N, a.Hkv, a.kd, BN)) return cudaErrorInvalidValue;
    tmV = tmQ;
    if (!a.emit_plane && !map_bnhx(&tmV, a.v, a.B, a.N, a.Hkv, D, BN)) return cudaErrorInvalidValue;
    tmY = tmQ;
    CUtensorMap tmC = tmQ;
    // Score planes are blocked [row block of 128][column block of 64][row in block][b*Hq + h][64 columns]: the 32
    // heads of a position lie 128 bytes apart (the aligner gathers them), and a head's 128 x 64 tile is 128 rows of 128
    // bytes spread over one 128 * B*Hq * 128-byte block, which the CTAs of all heads fill or drain at about the same time.
    if (a.emit_plane || a.plane) {
        if (a.plane_rows % BM != 0 || a.plane_cols % BN != 0) return cudaErrorInvalidValue;
        const uint64_t bh = (uint64_t)a.B * a.Hq, ncb = (uint64_t)a.plane_cols / BN, nrb = (uint64_t)a.plane_rows / BM;
        const uint64_t dims[5] = {(uint64_t)BN, bh, (uint64_t)BM, ncb, nrb};
        const uint64_t str[4] = {(uint64_t)BN * 2, bh * BN * 2, (uint64_t)BM * bh * BN * 2, ncb * BM * bh * BN * 2};
        // emit: one epilogue warp's 32 rows x 64 columns per copy; attention: the CTA's 128 rows x 64 columns
        const uint32_t box[5] = {(uint32_t)BN, 1, a.emit_plane ? 32u : (uint32_t)BM, 1, 1};
        if (!make_tensor_map_bf16(&tmY, a.emit_plane ? a.emit_plane : a.plane, 5, dims, str, box, true)) return cudaErrorInvalidValue;
        if (a.carry) {   // the logits leave one softmax warp's 32 rows at a time
            if (a.emit_plane || !a.plane) return cudaErrorInvalidValue;
            const uint32_t cbox[5] = {(uint32_t)BN, 1, 32u, 1, 1};
            if (!make_tensor_map_bf16(&tmC, a.carry, 5, dims, str, cbox, true)) return cudaErrorInvalidValue;
        }
    }
    FlashParams p;
    p.B = a.B; p.N = a.N; p.Hq = a.Hq; p.Hkv = a.Hkv;
    p.scale_log2 = a.scale * 1.4426950408889634f;
    p.o = reinterpret_cast<__nv_bfloat16*>(a.o.ptr);
    p.o_sb = a.o.stride_b; p.o_sn = a.o.stride_n; p.o_sh = a.o.stride_h;
    p.status = status_words();
    if (!p.status) return cudaErrorUnknown;
    p.plane_row0 = a.plane_row0 >= 0 ? a.plane_row0 : a.qt_begin * BM;
    if (p.plane_row0 % BM != 0 || p.plane_row0 > a.qt_begin * BM) return cudaErrorInvalidValue;
    p.qt_begin = a.qt_begin;
    p.ksteps = a.ksteps > 0 ? a.ksteps : a.kd / 16;
    p.scale = a.scale;

    if (a.qt_count < 1 || a.qt_count > 65535) return cudaErrorInvalidValue;
    // (batch, head) pairs that the CTAs are handed out for one after the other, in groups whose K and V fit half of a 126 MB L2 (the other half for
    // everything else that streams), so that the ~300 CTAs resident at a time re-read them from there for every query tile.  All pairs where they
    // fit; else all divided by the smallest prime factor of the batch count until they do, sequence by sequence from there, then by those of the
    // heads: equal groups, so a batch of 13 goes from all at once to one sequence.  Larger ones are better, because the heads of a position lie side
    // by side in a plane, whose lines the CTAs of neighbouring heads then write at about the same time, and because a grid ends with the lightest
    // tiles of its last group only.  One pair at a time, as it was beyond 63 MB | this, us: write-back at 4 x 8192 tokens of 32 / 8 heads
    // 4171 | 3452, 2 x 4096 of 32 / 32 heads 509 | 434, attention over 2 x 1777 of 40 heads 109 | 88; an anchor and one carried layer, prime
    // batches: 13 x 2048 of 32 / 8 heads 2552 | 2496, 61 x 1200 4997 | 4813, 7 x 1500 of 40 heads 1201 | 1157.
    const int64_t kv_head = (int64_t)a.N * (a.kd + (a.emit_plane ? 0 : D)) * 2;
    int group = a.B * a.Hq;
    if (a.qt_count > 1)
        while (group > 1 && ((group + a.Hq / a.Hkv - 1) / (a.Hq / a.Hkv)) * kv_head > ((int64_t)63 << 20)) {
            int d = 2;   // smallest factor: batches first, then heads
            const int over = group > a.Hq ? group / a.Hq : group;
            while (over % d) ++d;
            group /= d;
        }
    if (a.B * a.Hq / group > 65535) group = a.B * a.Hq;
    const dim3 grid(group, a.qt_count, a.B * a.Hq / group);
    cudaError_t e;
#define LISA_LAUNCH_FLASH(KD_, PL_)                                                                                       \
    do {                                                                                                                   \
        auto kern = tc_flash_kernel<KD_, PL_>;                                                                             \
        if ((e = allow_smem(kern, Smem<KD_, PL_>::TOTAL, true)) != cudaSuccess) return e;                                  \
        e = launch_kernel(a.chained, kern, grid, dim3(kThreads), Smem<KD_, PL_>::TOTAL, stream, p, tmQ, tmK, tmV, tmY, tmC); \
    } while (0)
    if (a.emit_plane) {
        if (a.kd == 128) LISA_LAUNCH_FLASH(128, MODE_EMIT);
        else LISA_LAUNCH_FLASH(32, MODE_EMIT);
    } else if (a.kd == 128 && !a.plane) LISA_LAUNCH_FLASH(128, MODE_ATTN);
    else if (a.kd == 32 && a.plane && a.carry) LISA_LAUNCH_FLASH(32, MODE_ATTN_CARRY);
    else if (a.kd == 32 && a.plane) LISA_LAUNCH_FLASH(32, MODE_ATTN_PLANE);
    else return cudaErrorInvalidValue;  // 128-wide scores plus a plane do not fit shared memory
#undef LISA_LAUNCH_FLASH
    count_launches(1);
    return e;
}

}  // namespace lisa
