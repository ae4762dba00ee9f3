// Main attention kernel and Split-K reduction kernel for sm_100a (paper Section 4: "Native CUDA
// catalog"; Section 2.3 data-compute pipeline; Section 4.3 Split-K).
//
// One persistent CTA per SM walks the ordered work-item list.  Inside a CTA the roles are
// warp-specialised:
//   warps 0-3  softmax / correction / epilogue: one thread per query row (TMEM lane), reads the
//              score tile S from tensor memory, applies the intra-tile membership mask, keeps the
//              online-softmax state (m, l) in registers, writes bf16 P back into tensor memory;
//   warp 4     TMA producer: gathers K and V tiles by tile index into shared-memory rings
//              (128-byte swizzle), and the Q tile once per work item;
//   warp 5     MMA issuer: tcgen05.mma S = Q K^T (both operands in shared memory) and
//              O += P V (P from tensor memory, V from shared memory, MN-major), fp32 accumulators
//              in tensor memory; tcgen05.commit signals the mbarriers.
// S is double-buffered so Q K^T of tile j+1 overlaps the softmax of tile j.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

#include <atomic>

#include "bsa_common.h"
#include "sm100_ptx.cuh"

namespace bsa {

using namespace ptx;


// Optional timeline tracing (compile with -DBSA_TRACE): CTA 0 records clock64() at barrier events of the
// single-tile kernel, per role, into a device buffer that bsa_debug_trace_copy() reads back.
#if defined(BSA_TRACE) || defined(BSA_PHASES)
__device__ long long g_trace[12][4096];  // producer, Q K^T (or single) issuer, softmax warps 0-7, P V issuer (role 6 in the 7-warp kernel)
__device__ long long g_trace_aux[12][4];  // last tile's stamps inside softmax_tile, per warp
__device__ long long g_cta_times[2][4096];  // %globaltimer at entry and exit of every CTA of the ping-pong kernel
#endif
#ifdef BSA_TRACE
#define BSA_TRACE_DECL(n) int n = 0
#define BSA_TRACE_POINT(role, n, tag)                                              \
    do {                                                                           \
        if (blockIdx.x == 0 && (n) < 4096) g_trace[role][(n)++] = (clock64() << 8) | (tag); \
    } while (0)
#else
#define BSA_TRACE_DECL(n)
#define BSA_TRACE_POINT(role, n, tag)
#endif

// Optional phase accounting (compile with -DBSA_PHASES): every softmax warp of the ping-pong kernel adds up the clocks it
// spends between fixed points of its tile loop; CTA 1 writes the sums out at its end (bsa_debug_trace_copy, roles 2-9).
#ifdef BSA_PHASES
#define BSA_PH_DECL uint32_t ph_acc[8] = {0, 0, 0, 0, 0, 0, 0, 0}, ph_n = 0, ph_t = (uint32_t)clock()
#define BSA_PH(k) do { const uint32_t now_ = (uint32_t)clock(); ph_acc[k] += now_ - ph_t; ph_t = now_; } while (0)
#define BSA_STAMP(role, tile, k) do { if (blockIdx.x == 1 && (tile) >= 40 && (tile) < 240) g_trace[role][16 + 4 * ((tile) - 40) + (k)] = clock64(); } while (0)
#else
#define BSA_PH_DECL
#define BSA_PH(k)
#define BSA_STAMP(role, tile, k)
#endif

// Test hook (bsa_debug_withhold_arrival): while non-zero, the V producer of the ping-pong kernel leaves out the copy
// of the first tile of its CTA together with the arrival that would announce it.  Nothing is in flight for that slot,
// so nothing can fault; the waits that depend on the tile simply run out, which is how the give-up path (status word,
// copies in flight allowed to land, TMEM freed, kernel returns) is exercised without a protocol error.
__device__ int g_withhold_arrival = 0;

namespace {

constexpr int kMaxStages = 6;
constexpr int kThreads = 192;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColS0 = 0, kColS1 = 128, kColO = 256;
constexpr uint32_t kColP0 = 384, kColP1 = 448;  // separate bf16 P buffers of the column-split kernel
constexpr float kRescaleThreshold = 8.0f;  // log2 units: P stays below 2^8 between rescales

struct AttnParams {
    const WorkItem* items;
    const int32_t* tile_col;
    const uint64_t* tile_member;
    PlanCountersDev* counters;
    __nv_bfloat16* O;
    float* LSE;
    float* ws_O;
    float* ws_LSE;
    unsigned long long full_member;
    int64_t o_head, o_row;  // element strides of O (and of Q) between heads and between token rows
    int32_t o_wide;         // O lies on a 32-byte boundary (16 bytes are all that the caller promises)
    int32_t N;    // query tokens per head
    int32_t Nkv;  // key/value tokens per head
    int32_t lgBQ;   // log2(B_Q) when B_Q < 128, else 31 (row >> 31 == 0)
    int32_t lgBKV;  // log2(B_KV) when B_KV < T_KV, else 31
    int32_t sK, lgSK;  // logical KV sub-blocks per entry of the tile list, and its logarithm
    int32_t stages;    // K ring depth (and V ring depth for the single-tile kernel)
    int32_t stages_v;  // V ring depth of the paired kernel
    float scale_log2;  // log2(e) / sqrt(d)
};

struct __align__(8) Barriers {
    uint64_t q_full, q_empty, o_free;
    uint64_t k_full[kMaxStages], k_empty[kMaxStages], v_full[kMaxStages], v_empty[kMaxStages];
    uint64_t s_full[2], p_ready[2], pv_done[2];
};

// One score tile of one query row (thread = row = TMEM lane): mask, running reference maximum,
// P = exp2(s * c2 - m_ref) rounded to bf16 and written to t_p (over S in place when t_p == t_s), running sum.
// The reference maximum moves only when the tile maximum exceeds it by kRescaleThreshold (log2
// units), so P stays below 2^8 and the running output needs rescaling (by `alpha`) only then.
template <int TK, bool F16 = false>
__device__ __forceinline__ void softmax_tile(uint32_t t_s, uint32_t t_p, bool need_mask, uint32_t row_bits, int lgBKV, int n_valid,
                                             float c2, bool not_first, float& m_ref, float& l, float& alpha,
                                             bool& rescale) {
    uint32_t r[TK];
#pragma unroll
    for (int c = 0; c < TK / 32; ++c) tmem_ld32(t_s + c * 32, &r[c * 32]);
    tc_wait_ld();
#ifdef BSA_TRACE
    if ((threadIdx.x & 31) == 0 && blockIdx.x == 0) g_trace_aux[threadIdx.x >> 5][0] = clock64();
#endif
    if (need_mask) {
        // B_KV >= 16: a group of 16 key columns lies inside one logical block, so one activity bit serves the group
#pragma unroll
        for (int gq = 0; gq < TK / 16; ++gq) {
            const bool grp = (row_bits >> ((gq * 16) >> lgBKV)) & 1u;
#pragma unroll
            for (int i = gq * 16; i < gq * 16 + 16; ++i) r[i] = (grp && i < n_valid) ? r[i] : 0xff800000u;  // -inf
        }
    }
    float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
    for (int i = 0; i < TK; i += 8) {
        m0 = max3(m0, __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
        m1 = max3(m1, __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3]));
        m2 = max3(m2, __uint_as_float(r[i + 4]), __uint_as_float(r[i + 5]));
        m3 = max3(m3, __uint_as_float(r[i + 6]), __uint_as_float(r[i + 7]));
    }
    const float mx2 = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3)) * c2;
    alpha = 1.f;
    rescale = false;
    if (mx2 > m_ref + kRescaleThreshold) {
        alpha = ex2_approx(m_ref - mx2);  // m_ref = -inf -> 0
        rescale = not_first && (m_ref != -INFINITY);
        m_ref = mx2;
    }
    const float neg_m = (m_ref == -INFINITY) ? 0.f : -m_ref;
#ifdef BSA_TRACE
    if ((threadIdx.x & 31) == 0 && blockIdx.x == 0) g_trace_aux[threadIdx.x >> 5][1] = clock64();
#endif
    // scale-and-shift and the row sums run as packed two-lane fp32 operations
    const uint64_t c22 = pack_f32x2(c2, c2), nm2 = pack_f32x2(neg_m, neg_m);
    uint64_t sum01 = pack_f32x2(0.f, 0.f), sum23 = sum01;
#pragma unroll
    for (int i = 0; i < TK; i += 4) {
        float x0, x1, x2, x3;
        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), c22, nm2), x0, x1);
        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(r[i + 2]), __uint_as_float(r[i + 3])), c22, nm2), x2, x3);
        const float p0 = ex2_approx(x0), p1 = ex2_approx(x1), p2 = ex2_approx(x2), p3 = ex2_approx(x3);
        sum01 = add_f32x2(sum01, pack_f32x2(p0, p1));
        sum23 = add_f32x2(sum23, pack_f32x2(p2, p3));
        r[i / 2] = pack_16x2<F16>(p0, p1);
        r[i / 2 + 1] = pack_16x2<F16>(p2, p3);
    }
    float s0, s1, s2, s3;
    unpack_f32x2(sum01, s0, s1);
    unpack_f32x2(sum23, s2, s3);
#ifdef BSA_TRACE
    if ((threadIdx.x & 31) == 0 && blockIdx.x == 0) g_trace_aux[threadIdx.x >> 5][2] = clock64();
#endif
#pragma unroll
    for (int c = 0; c < TK / 32; ++c) tmem_st16(t_p + c * 16, &r[c * 16]);
    l = l * alpha + ((s0 + s1) + (s2 + s3));
}

// DUAL = true adds a seventh warp so that Q K^T and P V are issued by two different threads: the
// Q K^T issuer runs up to two tiles ahead (S is double-buffered) instead of stalling behind the wait
// for the softmax of the previous tile; ordering between the two issuers is carried by mbarriers only.
template <int D, int TK, bool DUAL, bool F16>
__global__ void __launch_bounds__(DUAL ? kThreads + 32 : kThreads, 1)
bsa_attention_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                     const __grid_constant__ CUtensorMap tmV, const AttnParams p) {
    constexpr int NSUB = D / 64;              // 64-column (128-byte) sub-tiles per row
    constexpr int Q_SUB = kTQ * 128;          // bytes of one [128][64] bf16 sub-tile
    constexpr int KV_SUB = TK * 128;          // bytes of one [TK][64] bf16 sub-tile
    constexpr int KV_TILE = NSUB * KV_SUB;
    // dynamic shared memory starts on a 1024-byte boundary (the swizzled tiles need it); checked below
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sQ = smem;
    uint8_t* sK = sQ + NSUB * Q_SUB;
    uint8_t* sV = sK + p.stages * KV_TILE;
    __shared__ Barriers bars;
    __shared__ uint32_t tmem_base_s;
    __shared__ uint32_t abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (smem_u32(smem) & 1023u) {  // never expected; fail with a status instead of corrupting tiles
        if (tid == 0) atomicExch(&p.counters->status, (int)BSA_ERR_CUDA);
        return;
    }
    const int NS = p.stages;

    if (tid == 0) {
        abort_flag = 0;
        mbar_init(smem_u32(&bars.q_full), 1);
        mbar_init(smem_u32(&bars.q_empty), 1);
        mbar_init(smem_u32(&bars.o_free), 128);
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(smem_u32(&bars.k_full[s]), 1);
            mbar_init(smem_u32(&bars.k_empty[s]), 1);
            mbar_init(smem_u32(&bars.v_full[s]), 1);
            mbar_init(smem_u32(&bars.v_empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bars.s_full[s]), 1);
            mbar_init(smem_u32(&bars.p_ready[s]), 128);
            mbar_init(smem_u32(&bars.pv_done[s]), 1);
        }
        fence_mbar_init();
    }
    if (warp == 5) {
        tmem_alloc(smem_u32(&tmem_base_s), kTmemCols);
        tmem_relinquish();
    }
    if (warp == 4 && lane == 0) {
        prefetch_tensormap(&tmQ);
        prefetch_tensormap(&tmK);
        prefetch_tensormap(&tmV);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    volatile uint32_t* abortp = &abort_flag;
    const int n_items = p.counters->nitems;

    if (warp == 4) {
        // =========================== TMA producer ===========================
        if (lane == 0) {
            uint32_t itq = 0, g = 0;
            bool ok = true;
            BSA_TRACE_DECL(tn);
            for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
                const WorkItem it = p.items[idx];
                if (it.ntiles == 0) continue;
                ok = mbar_wait(smem_u32(&bars.q_empty), (itq & 1) ^ 1, abortp);
                if (!ok) break;
                mbar_arrive_expect_tx(smem_u32(&bars.q_full), NSUB * Q_SUB);
                for (int s = 0; s < NSUB; ++s)
                    tma_load_3d(smem_u32(sQ + s * Q_SUB), &tmQ, smem_u32(&bars.q_full), s * 64, it.q_tile * kTQ, it.head);
                int col_next = p.tile_col[it.tile_begin];  // tile metadata is fetched one tile ahead of its use
                for (int j = it.tile_begin; j < it.tile_end; ++j, ++g) {
                    const int col_cur = col_next;
                    if (j + 1 < it.tile_end) col_next = p.tile_col[j + 1];
                    const int stage = g % NS;
                    const uint32_t ph = (g / NS) & 1;
                    const int kv0 = col_cur * TK;
                    ok = mbar_wait(smem_u32(&bars.k_empty[stage]), ph ^ 1, abortp);
                    if (!ok) break;
                    BSA_TRACE_POINT(0, tn, 20);
                    mbar_arrive_expect_tx(smem_u32(&bars.k_full[stage]), KV_TILE);
                    for (int s = 0; s < NSUB; ++s)
                        tma_load_3d(smem_u32(sK + stage * KV_TILE + s * KV_SUB), &tmK, smem_u32(&bars.k_full[stage]),
                                    s * 64, kv0, it.head);
                    ok = mbar_wait(smem_u32(&bars.v_empty[stage]), ph ^ 1, abortp);
                    if (!ok) break;
                    BSA_TRACE_POINT(0, tn, 22);
                    mbar_arrive_expect_tx(smem_u32(&bars.v_full[stage]), KV_TILE);
                    for (int s = 0; s < NSUB; ++s)
                        tma_load_3d(smem_u32(sV + stage * KV_TILE + s * KV_SUB), &tmV, smem_u32(&bars.v_full[stage]),
                                    s * 64, kv0, it.head);
                }
                ++itq;
            }
            if (!ok) {
                // let copies in flight land before the CTA's shared memory goes away
                const uint64_t t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
            }
        }
    } else if (warp == 5 && !DUAL) {
        // =========================== MMA issuer ===========================
        if (lane == 0) {
            constexpr uint32_t idesc_qk = make_idesc_f32(kTQ, TK, 0, 0, F16);
            constexpr uint32_t idesc_pv = make_idesc_f32(kTQ, D, 0, 1, F16);
            const uint64_t descQ = make_smem_desc_sw128(smem_u32(sQ), 16, 1024);
            const uint64_t descK = make_smem_desc_sw128(smem_u32(sK), 16, 1024);
            const uint64_t descV = make_smem_desc_sw128(smem_u32(sV), KV_SUB, 1024);
            uint32_t itq = 0, g = 0;
            bool ok = true;
            BSA_TRACE_DECL(tn);
            for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
                const int n = p.items[idx].ntiles;
                if (n == 0) continue;
                ok = mbar_wait(smem_u32(&bars.q_full), itq & 1, abortp);
                if (!ok) break;
                for (int j = 0; j <= n && ok; ++j) {
                    if (j < n) {
                        const uint32_t gs = g + j;
                        const int stage = gs % NS;
                        const uint32_t ph = (gs / NS) & 1, sb = gs & 1;
                        ok = mbar_wait(smem_u32(&bars.k_full[stage]), ph, abortp);
                        if (!ok) break;
                        BSA_TRACE_POINT(1, tn, 1);
                        tc_fence_after();
                        // S[sb] = Q K^T.  The previous user of S[sb] (P of tile gs-2, read by its PV MMA)
                        // precedes this MMA in issue order on the same pipe.
                        const uint32_t d_s = tmem + (sb ? kColS1 : kColS0);
#pragma unroll
                        for (int k = 0; k < D / 16; ++k) {
                            const uint64_t a = descQ + (uint64_t)(((k / 4) * Q_SUB + (k % 4) * 32) >> 4);
                            const uint64_t b = descK + (uint64_t)((stage * KV_TILE + (k / 4) * KV_SUB + (k % 4) * 32) >> 4);
                            mma_ss(d_s, a, b, idesc_qk, k > 0);
                        }
                        mma_commit(smem_u32(&bars.k_empty[stage]));
                        mma_commit(smem_u32(&bars.s_full[sb]));
                        BSA_TRACE_POINT(1, tn, 2);
                        if (j == n - 1) mma_commit(smem_u32(&bars.q_empty));
                    }
                    if (j >= 1) {
                        const uint32_t gp = g + j - 1;
                        const int stage = gp % NS;
                        const uint32_t ph = (gp / NS) & 1, sb = gp & 1;
                        ok = mbar_wait(smem_u32(&bars.p_ready[sb]), (gp >> 1) & 1, abortp);
                        if (!ok) break;
                        BSA_TRACE_POINT(1, tn, 3);
                        ok = mbar_wait(smem_u32(&bars.v_full[stage]), ph, abortp);
                        if (!ok) break;
                        BSA_TRACE_POINT(1, tn, 4);
                        if (j == 1) {
                            ok = mbar_wait(smem_u32(&bars.o_free), (itq & 1) ^ 1, abortp);
                            if (!ok) break;
                        }
                        tc_fence_after();
                        const uint32_t a_p = tmem + (sb ? kColS1 : kColS0);
#pragma unroll
                        for (int k = 0; k < TK / 16; ++k) {
                            const uint64_t b = descV + (uint64_t)((stage * KV_TILE + k * 2048) >> 4);
                            mma_ts(tmem + kColO, a_p + k * 8, b, idesc_pv, (j > 1 || k > 0) ? 1u : 0u);
                        }
                        mma_commit(smem_u32(&bars.v_empty[stage]));
                        mma_commit(smem_u32(&bars.pv_done[sb]));
                        BSA_TRACE_POINT(1, tn, 5);
                    }
                }
                g += n;
                ++itq;
            }
        }
    } else if (warp == 5) {
        // =========================== Q K^T issuer (DUAL) ===========================
        if (lane == 0) {
            constexpr uint32_t idesc_qk = make_idesc_f32(kTQ, TK, 0, 0, F16);
            const uint64_t descQ = make_smem_desc_sw128(smem_u32(sQ), 16, 1024);
            const uint64_t descK = make_smem_desc_sw128(smem_u32(sK), 16, 1024);
            uint32_t itq = 0, g = 0;
            bool ok = true;
            BSA_TRACE_DECL(tn);
            for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
                const int n = p.items[idx].ntiles;
                if (n == 0) continue;
                ok = mbar_wait(smem_u32(&bars.q_full), itq & 1, abortp);
                if (!ok) break;
                for (int j = 0; j < n; ++j) {
                    const uint32_t gs = g + j;
                    const int stage = gs % NS;
                    const uint32_t ph = (gs / NS) & 1, sb = gs & 1;
                    ok = mbar_wait(smem_u32(&bars.k_full[stage]), ph, abortp);
                    if (!ok) break;
                    BSA_TRACE_POINT(1, tn, 1);
                    // S[sb] still holds P of tile gs-2 (written in place) until that tile's P V has completed.
                    // (Measured: giving P its own columns so that Q K^T may start right after the softmax of
                    // tile gs-2 was slower -- the early Q K^T delays the P V the softmax chain is waiting for.)
                    if (gs >= 2) {
                        ok = mbar_wait(smem_u32(&bars.pv_done[sb]), ((gs >> 1) - 1) & 1, abortp);
                        if (!ok) break;
                    }
                    BSA_TRACE_POINT(1, tn, 6);
                    tc_fence_after();
                    const uint32_t d_s = tmem + (sb ? kColS1 : kColS0);
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) {
                        const uint64_t a = descQ + (uint64_t)(((k / 4) * Q_SUB + (k % 4) * 32) >> 4);
                        const uint64_t b = descK + (uint64_t)((stage * KV_TILE + (k / 4) * KV_SUB + (k % 4) * 32) >> 4);
                        mma_ss(d_s, a, b, idesc_qk, k > 0);
                    }
                    mma_commit(smem_u32(&bars.k_empty[stage]));
                    mma_commit(smem_u32(&bars.s_full[sb]));
                    BSA_TRACE_POINT(1, tn, 2);
                    if (j == n - 1) mma_commit(smem_u32(&bars.q_empty));
                }
                g += n;
                ++itq;
            }
        }
    } else if (warp == 6) {
        // =========================== P V issuer (DUAL) ===========================
        if (lane == 0) {
            constexpr uint32_t idesc_pv = make_idesc_f32(kTQ, D, 0, 1, F16);
            const uint64_t descV = make_smem_desc_sw128(smem_u32(sV), KV_SUB, 1024);
            uint32_t itq = 0, g = 0;
            bool ok = true;
            BSA_TRACE_DECL(tn);
            for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
                const int n = p.items[idx].ntiles;
                if (n == 0) continue;
                for (int j = 0; j < n; ++j) {
                    const uint32_t gp = g + j;
                    const int stage = gp % NS;
                    const uint32_t ph = (gp / NS) & 1, sb = gp & 1;
                    ok = mbar_wait(smem_u32(&bars.p_ready[sb]), (gp >> 1) & 1, abortp);
                    if (!ok) break;
                    BSA_TRACE_POINT(6, tn, 3);
                    ok = mbar_wait(smem_u32(&bars.v_full[stage]), ph, abortp);
                    if (!ok) break;
                    if (j == 0) {
                        ok = mbar_wait(smem_u32(&bars.o_free), (itq & 1) ^ 1, abortp);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    const uint32_t a_p = tmem + (sb ? kColS1 : kColS0);
#pragma unroll
                    for (int k = 0; k < TK / 16; ++k) {
                        const uint64_t b = descV + (uint64_t)((stage * KV_TILE + k * 2048) >> 4);
                        mma_ts(tmem + kColO, a_p + k * 8, b, idesc_pv, (j > 0 || k > 0) ? 1u : 0u);
                    }
                    mma_commit(smem_u32(&bars.v_empty[stage]));
                    mma_commit(smem_u32(&bars.pv_done[sb]));
                    BSA_TRACE_POINT(6, tn, 5);
                }
                g += n;
                ++itq;
            }
        }
    } else {
        // =========================== softmax / correction / epilogue ===========================
        const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
        uint32_t itq = 0, g = 0;
        bool ok = true;
        BSA_TRACE_DECL(tn);
        const float c2 = p.scale_log2;
        const unsigned long long sub_mask = (p.sK >= 64) ? ~0ull : ((1ull << p.sK) - 1ull);
        for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
            const WorkItem it = p.items[idx];
            const int row = it.q_tile * kTQ + tid;
            const bool row_ok = row < p.N;
            if (it.ntiles == 0) {
                // no physical tile touches this Q tile row: O = 0, LSE = -inf
                if (row_ok) {
                    uint4* o = reinterpret_cast<uint4*>(p.O + ((size_t)it.head * p.o_head + (size_t)row * p.o_row));
#pragma unroll
                    for (int c = 0; c < D / 8; ++c) o[c] = make_uint4(0, 0, 0, 0);
                    p.LSE[(size_t)it.head * p.N + row] = -INFINITY;
                }
                continue;
            }
            float m_ref = -INFINITY, l = 0.f;
            int col_next = p.tile_col[it.tile_begin];  // tile metadata is fetched one tile ahead of its use
            unsigned long long member_next = p.tile_member[it.tile_begin];
            for (int j = 0; j < it.ntiles; ++j) {
                const uint32_t gs = g + j, sb = gs & 1;
                const int kv0 = col_next * TK;
                const unsigned long long member = member_next;
                if (j + 1 < it.ntiles) {
                    col_next = p.tile_col[it.tile_begin + j + 1];
                    member_next = p.tile_member[it.tile_begin + j + 1];
                }
                const bool need_mask = (member != p.full_member) || (kv0 + TK > p.Nkv);
                const uint32_t row_bits = (uint32_t)((member >> ((tid >> p.lgBQ) * p.sK)) & sub_mask);
                const int n_valid = p.Nkv - kv0;  // columns >= n_valid do not exist
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.s_full[sb]), (gs >> 1) & 1, abortp));
                if (!ok) break;
                if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 10);
                tc_fence_after();
                const uint32_t t_s = tmem + lane_base + (sb ? kColS1 : kColS0);
                float alpha;
                bool rescale;
                softmax_tile<TK, F16>(t_s, t_s, need_mask, row_bits, p.lgBKV, n_valid, c2, j > 0, m_ref, l, alpha, rescale);
#ifdef BSA_TRACE
                if (lane == 0 && blockIdx.x == 0 && tn + 3 < 4096) {
                    g_trace[2 + warp][tn++] = (g_trace_aux[warp][0] << 8) | 11;
                    g_trace[2 + warp][tn++] = (g_trace_aux[warp][1] << 8) | 12;
                    g_trace[2 + warp][tn++] = (g_trace_aux[warp][2] << 8) | 14;
                }
#endif
                if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 13);
                // ---- correction: rescale the running output when the reference moved ----
                if (j > 0 && __any_sync(0xffffffffu, rescale)) {
                    const uint32_t gp = gs - 1;
                    ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.pv_done[gp & 1]), (gp >> 1) & 1, abortp));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t t_o = tmem + lane_base + kColO;
#pragma unroll
                    for (int c = 0; c < D / 32; ++c) {
                        uint32_t r[32];
                        tmem_ld32(t_o + c * 32, r);
                        tc_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
                        tmem_st32(t_o + c * 32, r);
                    }
                }
                tc_wait_st();
                tc_fence_before();
                mbar_arrive(smem_u32(&bars.p_ready[sb]));
                if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 16);
            }
            if (!ok) break;
            // ---- epilogue ----
            {
                const uint32_t gl = g + it.ntiles - 1;
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.pv_done[gl & 1]), (gl >> 1) & 1, abortp));
                if (!ok) break;
                tc_fence_after();
                const float inv_l = (l > 0.f) ? 1.f / l : 0.f;
                const float lse = (l > 0.f) ? fmaf(m_ref, 0.6931471805599453f, logf(l)) : -INFINITY;
                const uint32_t t_o = tmem + lane_base + kColO;
                if (it.nparts == 1) {
                    __nv_bfloat16* orow = p.O + ((size_t)it.head * p.o_head + (size_t)row * p.o_row);
#pragma unroll
                    for (int c = 0; c < D / 32; ++c) {
                        uint32_t r[32];
                        tmem_ld32(t_o + c * 32, r);
                        tc_wait_ld();
                        if (row_ok) {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                uint4 v;
                                v.x = pack_16x2<F16>(__uint_as_float(r[q * 8 + 0]) * inv_l, __uint_as_float(r[q * 8 + 1]) * inv_l);
                                v.y = pack_16x2<F16>(__uint_as_float(r[q * 8 + 2]) * inv_l, __uint_as_float(r[q * 8 + 3]) * inv_l);
                                v.z = pack_16x2<F16>(__uint_as_float(r[q * 8 + 4]) * inv_l, __uint_as_float(r[q * 8 + 5]) * inv_l);
                                v.w = pack_16x2<F16>(__uint_as_float(r[q * 8 + 6]) * inv_l, __uint_as_float(r[q * 8 + 7]) * inv_l);
                                *reinterpret_cast<uint4*>(orow + c * 32 + q * 8) = v;
                            }
                        }
                    }
                    if (row_ok) p.LSE[(size_t)it.head * p.N + row] = lse;
                } else {
                    float* orow = p.ws_O + ((size_t)it.ws_slot * kTQ + tid) * D;
#pragma unroll
                    for (int c = 0; c < D / 32; ++c) {
                        uint32_t r[32];
                        tmem_ld32(t_o + c * 32, r);
                        tc_wait_ld();
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            float4 v = make_float4(__uint_as_float(r[q * 4 + 0]) * inv_l, __uint_as_float(r[q * 4 + 1]) * inv_l,
                                                   __uint_as_float(r[q * 4 + 2]) * inv_l, __uint_as_float(r[q * 4 + 3]) * inv_l);
                            *reinterpret_cast<float4*>(orow + c * 32 + q * 4) = v;
                        }
                    }
                    p.ws_LSE[(size_t)it.ws_slot * kTQ + tid] = lse;
                }
                tc_fence_before();
                mbar_arrive(smem_u32(&bars.o_free));
            }
            g += it.ntiles;
            ++itq;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (tid == 0 && abort_flag) atomicExch(&p.counters->status, (int)BSA_ERR_DEVICE_TIMEOUT);
    if (warp == 5) tmem_dealloc(tmem, kTmemCols);
}

// ==========================================================================================
// Paired kernel: one CTA owns a 256-row physical Q tile as two 128-row MMA slots.  Both slots
// walk the same (merged) KV tile list, so every K/V tile is fetched into shared memory once and
// feeds up to two Q tiles; a slot whose membership word for a tile is zero skips it.  Each slot
// has its own softmax warpgroup, S/P columns and O accumulator in tensor memory; the single MMA
// warp alternates between the slots (PV of the previous tile, then Q K^T of the next), so one
// slot's softmax runs under the other slot's MMAs.
//   warps 0-3 / 4-7 : softmax + correction + epilogue of slot 0 / slot 1 (more registers)
//   warp 8          : TMA producer    warp 9 : Q K^T issuer    warp 10 : P V issuer (this warpgroup gives registers back)
// Register budget: 384 threads launch with 168 registers each (504 per lane across the three
// warpgroups); setmaxnreg moves them to 216 + 216 + 72 = 504.  The sum must not exceed the launch
// allocation, otherwise the second setmaxnreg.inc never gets its registers and the CTA stalls.
// ==========================================================================================
constexpr int kPairThreads = 384;

struct __align__(8) PairBarriers {
    uint64_t q_full, q_empty;
    uint64_t k_full[kMaxStages], k_empty[kMaxStages], v_full[kMaxStages], v_empty[kMaxStages];
    uint64_t s_full[2], p_ready[2], pv_done[2], o_free[2];
};

template <int R>
__device__ __forceinline__ void reg_inc() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R));
}
template <int R>
__device__ __forceinline__ void reg_dec() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R));
}

template <int D, int TK>
__global__ void __launch_bounds__(kPairThreads, 1)
bsa_attention_pair_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                          const __grid_constant__ CUtensorMap tmV, const AttnParams p) {
    constexpr int NSUB = D / 64;
    constexpr int Q_SUB = kTQ * 128;
    constexpr int Q_TILE = NSUB * Q_SUB;
    constexpr int KV_SUB = TK * 128;
    constexpr int KV_TILE = NSUB * KV_SUB;
    // dynamic shared memory starts on a 1024-byte boundary (the swizzled tiles need it); checked below
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sQ = smem;                       // [2 slots][NSUB][128][64]
    uint8_t* sK = sQ + 2 * Q_TILE;            // [stages][NSUB][TK][64]
    uint8_t* sV = sK + p.stages * KV_TILE;    // [stages_v][NSUB][TK][64]
    __shared__ PairBarriers bars;
    __shared__ uint32_t tmem_base_s;
    __shared__ uint32_t abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (smem_u32(smem) & 1023u) {  // never expected; fail with a status instead of corrupting tiles
        if (tid == 0) atomicExch(&p.counters->status, (int)BSA_ERR_CUDA);
        return;
    }
    const int NSK = p.stages, NSV = p.stages_v;

    if (tid == 0) {
        abort_flag = 0;
        mbar_init(smem_u32(&bars.q_full), 1);
        mbar_init(smem_u32(&bars.q_empty), 1);
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(smem_u32(&bars.k_full[s]), 1);
            mbar_init(smem_u32(&bars.k_empty[s]), 1);
            mbar_init(smem_u32(&bars.v_full[s]), 1);
            mbar_init(smem_u32(&bars.v_empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bars.s_full[s]), 1);
            mbar_init(smem_u32(&bars.p_ready[s]), 128);
            mbar_init(smem_u32(&bars.pv_done[s]), 1);
            mbar_init(smem_u32(&bars.o_free[s]), 128);
        }
        fence_mbar_init();
    }
    if (warp == 9) {
        tmem_alloc(smem_u32(&tmem_base_s), kTmemCols);
        tmem_relinquish();
    }
    if (warp == 8 && lane == 0) {
        prefetch_tensormap(&tmQ);
        prefetch_tensormap(&tmK);
        prefetch_tensormap(&tmV);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    volatile uint32_t* abortp = &abort_flag;
    const int n_items = p.counters->nitems;

    if (warp >= 8) {
        reg_dec<72>();
        if (warp == 8 && lane == 0) {
            // =========================== TMA producer ===========================
            uint32_t itq = 0, g = 0;
            bool ok = true;
            for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
                const WorkItem it = p.items[idx];
                if (it.ntiles == 0) continue;
                ok = mbar_wait(smem_u32(&bars.q_empty), (itq & 1) ^ 1, abortp);
                if (!ok) break;
                mbar_arrive_expect_tx(smem_u32(&bars.q_full), 2 * Q_TILE);
                for (int x = 0; x < 2; ++x)
                    for (int s = 0; s < NSUB; ++s)
                        tma_load_3d(smem_u32(sQ + x * Q_TILE + s * Q_SUB), &tmQ, smem_u32(&bars.q_full), s * 64,
                                    it.q_tile * (2 * kTQ) + x * kTQ, it.head);
                int col_next = p.tile_col[it.tile_begin];  // tile metadata is fetched one tile ahead of its use
                for (int j = it.tile_begin; j < it.tile_end; ++j, ++g) {
                    const int col_cur = col_next;
                    if (j + 1 < it.tile_end) col_next = p.tile_col[j + 1];
                    const int sk = g % NSK, sv = g % NSV;
                    const uint32_t phk = (g / NSK) & 1, phv = (g / NSV) & 1;
                    const int kv0 = col_cur * TK;
                    ok = mbar_wait(smem_u32(&bars.k_empty[sk]), phk ^ 1, abortp);
                    if (!ok) break;
                    mbar_arrive_expect_tx(smem_u32(&bars.k_full[sk]), KV_TILE);
                    for (int s = 0; s < NSUB; ++s)
                        tma_load_3d(smem_u32(sK + sk * KV_TILE + s * KV_SUB), &tmK, smem_u32(&bars.k_full[sk]), s * 64,
                                    kv0, it.head);
                    ok = mbar_wait(smem_u32(&bars.v_empty[sv]), phv ^ 1, abortp);
                    if (!ok) break;
                    mbar_arrive_expect_tx(smem_u32(&bars.v_full[sv]), KV_TILE);
                    for (int s = 0; s < NSUB; ++s)
                        tma_load_3d(smem_u32(sV + sv * KV_TILE + s * KV_SUB), &tmV, smem_u32(&bars.v_full[sv]), s * 64,
                                    kv0, it.head);
                }
                ++itq;
            }
            if (!ok) {
                const uint64_t t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
            }
        } else if (warp == 9 && lane == 0) {
            // =========================== Q K^T issuer (both slots) ===========================
            constexpr uint32_t idesc_qk = make_idesc_bf16_f32(kTQ, TK, 0, 0);
            const uint64_t descQ = make_smem_desc_sw128(smem_u32(sQ), 16, 1024);
            const uint64_t descK = make_smem_desc_sw128(smem_u32(sK), 16, 1024);
            uint32_t itq = 0, g = 0;
            uint32_t nqk[2] = {0, 0};  // Q K^T tiles issued per slot
            bool ok = true;
            for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
                const WorkItem it = p.items[idx];
                const int n = it.ntiles;
                if (n == 0) continue;
                ok = mbar_wait(smem_u32(&bars.q_full), itq & 1, abortp);
                if (!ok) break;
                ulonglong2 mem_next = *reinterpret_cast<const ulonglong2*>(p.tile_member + (size_t)it.tile_begin * 2);
                for (int j = 0; j < n && ok; ++j) {
                    const uint32_t gj = g + j;
                    const int sk = gj % NSK;
                    const ulonglong2 mem = mem_next;
                    if (j + 1 < n)
                        mem_next = *reinterpret_cast<const ulonglong2*>(p.tile_member + (size_t)(it.tile_begin + j + 1) * 2);
                    ok = mbar_wait(smem_u32(&bars.k_full[sk]), (gj / NSK) & 1, abortp);
                    if (!ok) break;
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        if ((x == 0 ? mem.x : mem.y) == 0ull) continue;
                        // S_x holds the bf16 P of the slot's previous tile until that tile's P V has completed
                        if (nqk[x] >= 1) {
                            ok = mbar_wait(smem_u32(&bars.pv_done[x]), (nqk[x] - 1) & 1, abortp);
                            if (!ok) break;
                        }
                        tc_fence_after();
                        const uint32_t d_s = tmem + x * 128;
#pragma unroll
                        for (int k = 0; k < D / 16; ++k) {
                            const uint64_t a = descQ + (uint64_t)((x * Q_TILE + (k / 4) * Q_SUB + (k % 4) * 32) >> 4);
                            const uint64_t b = descK + (uint64_t)((sk * KV_TILE + (k / 4) * KV_SUB + (k % 4) * 32) >> 4);
                            mma_ss(d_s, a, b, idesc_qk, k > 0);
                        }
                        mma_commit(smem_u32(&bars.s_full[x]));
                        ++nqk[x];
                    }
                    if (!ok) break;
                    mma_commit(smem_u32(&bars.k_empty[sk]));
                }
                if (!ok) break;
                mma_commit(smem_u32(&bars.q_empty));
                g += n;
                ++itq;
            }
        } else if (warp == 10 && lane == 0) {
            // =========================== P V issuer (both slots) ===========================
            constexpr uint32_t idesc_pv = make_idesc_bf16_f32(kTQ, D, 0, 1);
            const uint64_t descV = make_smem_desc_sw128(smem_u32(sV), KV_SUB, 1024);
            uint32_t g = 0;
            uint32_t npv[2] = {0, 0};  // P V tiles issued per slot: phase of p_ready / pv_done
            uint32_t oit[2] = {0, 0};  // items in which the slot had tiles: phase of o_free
            bool ok = true;
            for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
                const WorkItem it = p.items[idx];
                const int n = it.ntiles;
                if (n == 0) continue;
                bool started[2] = {false, false};
                ulonglong2 mem_next = *reinterpret_cast<const ulonglong2*>(p.tile_member + (size_t)it.tile_begin * 2);
                for (int j = 0; j < n && ok; ++j) {
                    const uint32_t gj = g + j;
                    const int sv = gj % NSV;
                    const ulonglong2 mem = mem_next;
                    if (j + 1 < n)
                        mem_next = *reinterpret_cast<const ulonglong2*>(p.tile_member + (size_t)(it.tile_begin + j + 1) * 2);
                    ok = mbar_wait(smem_u32(&bars.v_full[sv]), (gj / NSV) & 1, abortp);
                    if (!ok) break;
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        if ((x == 0 ? mem.x : mem.y) == 0ull) continue;
                        ok = mbar_wait(smem_u32(&bars.p_ready[x]), npv[x] & 1, abortp);
                        if (!ok) break;
                        if (!started[x]) {
                            ok = mbar_wait(smem_u32(&bars.o_free[x]), (oit[x] & 1) ^ 1, abortp);
                            if (!ok) break;
                        }
                        tc_fence_after();
                        const uint32_t d_o = tmem + kColO + x * 128, a_p = tmem + x * 128;
#pragma unroll
                        for (int k = 0; k < TK / 16; ++k) {
                            const uint64_t b = descV + (uint64_t)((sv * KV_TILE + k * 2048) >> 4);
                            mma_ts(d_o, a_p + k * 8, b, idesc_pv, (started[x] || k > 0) ? 1u : 0u);
                        }
                        mma_commit(smem_u32(&bars.pv_done[x]));
                        ++npv[x];
                        started[x] = true;
                    }
                    if (!ok) break;
                    mma_commit(smem_u32(&bars.v_empty[sv]));
                }
                if (!ok) break;
                for (int x = 0; x < 2; ++x)
                    if (started[x]) ++oit[x];
                g += n;
            }
        }
    } else {
        // =========================== softmax / correction / epilogue of slot x ===========================
        reg_inc<216>();
        const int x = warp >> 2;
        const int tw = tid & 127;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t t_s = tmem + lane_base + x * 128;
        const uint32_t t_o = tmem + lane_base + kColO + x * 128;
        uint32_t cnt = 0;  // tiles this slot has processed: phase of s_full / p_ready / pv_done
        bool ok = true;
        const float c2 = p.scale_log2;
        const unsigned long long sub_mask = (p.sK >= 64) ? ~0ull : ((1ull << p.sK) - 1ull);
        for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
            const WorkItem it = p.items[idx];
            const int row = it.q_tile * (2 * kTQ) + x * kTQ + tw;
            const bool row_ok = row < p.N;
            float m_ref = -INFINITY, l = 0.f;
            int nmine = 0;
            int col_next = 0;
            unsigned long long member_next = 0ull;
            if (it.ntiles > 0) {  // tile metadata is fetched one tile ahead of its use
                col_next = p.tile_col[it.tile_begin];
                member_next = p.tile_member[(size_t)it.tile_begin * 2 + x];
            }
            for (int j = 0; j < it.ntiles; ++j) {
                const unsigned long long member = member_next;
                const int kv0 = col_next * TK;
                if (j + 1 < it.ntiles) {
                    col_next = p.tile_col[it.tile_begin + j + 1];
                    member_next = p.tile_member[(size_t)(it.tile_begin + j + 1) * 2 + x];
                }
                if (member == 0ull) continue;
                const bool need_mask = (member != p.full_member) || (kv0 + TK > p.Nkv);
                const uint32_t row_bits = (uint32_t)((member >> ((tw >> p.lgBQ) * p.sK)) & sub_mask);
                const int n_valid = p.Nkv - kv0;
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.s_full[x]), cnt & 1, abortp));
                if (!ok) break;
                tc_fence_after();
                float alpha;
                bool rescale;
                softmax_tile<TK>(t_s, t_s, need_mask, row_bits, p.lgBKV, n_valid, c2, nmine > 0, m_ref, l, alpha, rescale);
                if (nmine > 0 && __any_sync(0xffffffffu, rescale)) {
                    ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.pv_done[x]), (cnt - 1) & 1, abortp));
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int c = 0; c < D / 32; ++c) {
                        uint32_t r[32];
                        tmem_ld32(t_o + c * 32, r);
                        tc_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
                        tmem_st32(t_o + c * 32, r);
                    }
                }
                tc_wait_st();
                tc_fence_before();
                mbar_arrive(smem_u32(&bars.p_ready[x]));
                ++cnt;
                ++nmine;
            }
            if (!ok) break;
            if (nmine == 0) {
                // no tile of this item reaches this slot's rows: O = 0, LSE = -inf (or an empty partial state)
                if (it.nparts == 1) {
                    if (row_ok) {
                        uint4* o = reinterpret_cast<uint4*>(p.O + ((size_t)it.head * p.o_head + (size_t)row * p.o_row));
#pragma unroll
                        for (int c = 0; c < D / 8; ++c) o[c] = make_uint4(0, 0, 0, 0);
                        p.LSE[(size_t)it.head * p.N + row] = -INFINITY;
                    }
                } else {
                    float4* o = reinterpret_cast<float4*>(p.ws_O + ((size_t)(it.ws_slot + x) * kTQ + tw) * D);
#pragma unroll
                    for (int c = 0; c < D / 4; ++c) o[c] = make_float4(0.f, 0.f, 0.f, 0.f);
                    p.ws_LSE[(size_t)(it.ws_slot + x) * kTQ + tw] = -INFINITY;
                }
                continue;
            }
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.pv_done[x]), (cnt - 1) & 1, abortp));
            if (!ok) break;
            tc_fence_after();
            const float inv_l = (l > 0.f) ? 1.f / l : 0.f;
            const float lse = (l > 0.f) ? fmaf(m_ref, 0.6931471805599453f, logf(l)) : -INFINITY;
            if (it.nparts == 1) {
                __nv_bfloat16* orow = p.O + ((size_t)it.head * p.o_head + (size_t)row * p.o_row);
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t r[32];
                    tmem_ld32(t_o + c * 32, r);
                    tc_wait_ld();
                    if (row_ok) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            uint4 v;
                            v.x = pack_bf16x2(__uint_as_float(r[q * 8 + 0]) * inv_l, __uint_as_float(r[q * 8 + 1]) * inv_l);
                            v.y = pack_bf16x2(__uint_as_float(r[q * 8 + 2]) * inv_l, __uint_as_float(r[q * 8 + 3]) * inv_l);
                            v.z = pack_bf16x2(__uint_as_float(r[q * 8 + 4]) * inv_l, __uint_as_float(r[q * 8 + 5]) * inv_l);
                            v.w = pack_bf16x2(__uint_as_float(r[q * 8 + 6]) * inv_l, __uint_as_float(r[q * 8 + 7]) * inv_l);
                            *reinterpret_cast<uint4*>(orow + c * 32 + q * 8) = v;
                        }
                    }
                }
                if (row_ok) p.LSE[(size_t)it.head * p.N + row] = lse;
            } else {
                float* orow = p.ws_O + ((size_t)(it.ws_slot + x) * kTQ + tw) * D;
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t r[32];
                    tmem_ld32(t_o + c * 32, r);
                    tc_wait_ld();
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        float4 v = make_float4(__uint_as_float(r[q * 4 + 0]) * inv_l, __uint_as_float(r[q * 4 + 1]) * inv_l,
                                               __uint_as_float(r[q * 4 + 2]) * inv_l, __uint_as_float(r[q * 4 + 3]) * inv_l);
                        *reinterpret_cast<float4*>(orow + c * 32 + q * 4) = v;
                    }
                }
                p.ws_LSE[(size_t)(it.ws_slot + x) * kTQ + tw] = lse;
            }
            tc_fence_before();
            mbar_arrive(smem_u32(&bars.o_free[x]));
        }
    }

    tc_fence_before();
    __syncthreads();
    if (tid == 0 && abort_flag) atomicExch(&p.counters->status, (int)BSA_ERR_DEVICE_TIMEOUT);
    if (warp == 9) tmem_dealloc(tmem, kTmemCols);
}

// ==========================================================================================
// Column-split kernel: same work decomposition as bsa_attention_kernel (one 128-row Q tile per
// CTA, S double-buffered), but TWO threads per query row: softmax warps 0-3 take the left half of
// the score tile's columns, warps 4-7 the right half (both may read the same TMEM lanes).  The two
// threads of a row exchange their half-row maxima through shared memory so they take identical
// reference-maximum decisions; each keeps a partial sum, added up once in the epilogue.  P goes to
// its own TMEM columns (the halves of S being read by the partner must not be overwritten).
//   warps 0-7 : softmax / correction / epilogue    warp 8 : TMA producer
//   warp 9 : Q K^T issuer    warp 10 : P V issuer (separate threads, ordered through mbarriers only)
// ==========================================================================================
constexpr int kCsThreads = 352;

struct __align__(8) CsBarriers {
    uint64_t q_full, q_empty, o_free, xchg;
    uint64_t k_full[kMaxStages], k_empty[kMaxStages], v_full[kMaxStages], v_empty[kMaxStages];
    uint64_t s_full[2], p_ready[2], pv_done[2];
};

template <int D, int TK>
__global__ void __launch_bounds__(kCsThreads, 1)
bsa_attention_cs_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const AttnParams p) {
    constexpr int NSUB = D / 64;
    constexpr int Q_SUB = kTQ * 128;
    constexpr int KV_SUB = TK * 128;
    constexpr int KV_TILE = NSUB * KV_SUB;
    constexpr int NC = TK / 2;  // score columns per softmax thread
    constexpr int DC = D / 2;   // output columns per softmax thread
    // dynamic shared memory starts on a 1024-byte boundary (the swizzled tiles need it); checked below
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sQ = smem;
    uint8_t* sK = sQ + NSUB * Q_SUB;
    uint8_t* sV = sK + p.stages * KV_TILE;
    __shared__ CsBarriers bars;
    __shared__ float xbuf[2][2][kTQ];  // [use parity][column half][row]: half-row maxima / partial sums
    __shared__ uint32_t tmem_base_s;
    __shared__ uint32_t abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (smem_u32(smem) & 1023u) {  // never expected; fail with a status instead of corrupting tiles
        if (tid == 0) atomicExch(&p.counters->status, (int)BSA_ERR_CUDA);
        return;
    }
    const int NS = p.stages;

    if (tid == 0) {
        abort_flag = 0;
        mbar_init(smem_u32(&bars.q_full), 1);
        mbar_init(smem_u32(&bars.q_empty), 1);
        mbar_init(smem_u32(&bars.o_free), 256);
        mbar_init(smem_u32(&bars.xchg), 256);
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(smem_u32(&bars.k_full[s]), 1);
            mbar_init(smem_u32(&bars.k_empty[s]), 1);
            mbar_init(smem_u32(&bars.v_full[s]), 1);
            mbar_init(smem_u32(&bars.v_empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bars.s_full[s]), 1);
            mbar_init(smem_u32(&bars.p_ready[s]), 256);
            mbar_init(smem_u32(&bars.pv_done[s]), 1);
        }
        fence_mbar_init();
    }
    if (warp == 9) {
        tmem_alloc(smem_u32(&tmem_base_s), kTmemCols);
        tmem_relinquish();
    }
    if (warp == 8 && lane == 0) {
        prefetch_tensormap(&tmQ);
        prefetch_tensormap(&tmK);
        prefetch_tensormap(&tmV);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    volatile uint32_t* abortp = &abort_flag;
    const int n_items = p.counters->nitems;

    if (warp == 8) {
        // =========================== TMA producer ===========================
        if (lane == 0) {
            uint32_t itq = 0, g = 0;
            bool ok = true;
            for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
                const WorkItem it = p.items[idx];
                if (it.ntiles == 0) continue;
                ok = mbar_wait(smem_u32(&bars.q_empty), (itq & 1) ^ 1, abortp);
                if (!ok) break;
                mbar_arrive_expect_tx(smem_u32(&bars.q_full), NSUB * Q_SUB);
                for (int s = 0; s < NSUB; ++s)
                    tma_load_3d(smem_u32(sQ + s * Q_SUB), &tmQ, smem_u32(&bars.q_full), s * 64, it.q_tile * kTQ, it.head);
                int col_next = p.tile_col[it.tile_begin];  // tile metadata is fetched one tile ahead of its use
                for (int j = it.tile_begin; j < it.tile_end; ++j, ++g) {
                    const int col_cur = col_next;
                    if (j + 1 < it.tile_end) col_next = p.tile_col[j + 1];
                    const int stage = g % NS;
                    const uint32_t ph = (g / NS) & 1;
                    const int kv0 = col_cur * TK;
                    ok = mbar_wait(smem_u32(&bars.k_empty[stage]), ph ^ 1, abortp);
                    if (!ok) break;
                    mbar_arrive_expect_tx(smem_u32(&bars.k_full[stage]), KV_TILE);
                    for (int s = 0; s < NSUB; ++s)
                        tma_load_3d(smem_u32(sK + stage * KV_TILE + s * KV_SUB), &tmK, smem_u32(&bars.k_full[stage]),
                                    s * 64, kv0, it.head);
                    ok = mbar_wait(smem_u32(&bars.v_empty[stage]), ph ^ 1, abortp);
                    if (!ok) break;
                    mbar_arrive_expect_tx(smem_u32(&bars.v_full[stage]), KV_TILE);
                    for (int s = 0; s < NSUB; ++s)
                        tma_load_3d(smem_u32(sV + stage * KV_TILE + s * KV_SUB), &tmV, smem_u32(&bars.v_full[stage]),
                                    s * 64, kv0, it.head);
                }
                ++itq;
            }
            if (!ok) {
                const uint64_t t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
            }
        }
    } else if (warp == 9) {
        // =========================== Q K^T issuer ===========================
        if (lane == 0) {
            constexpr uint32_t idesc_qk = make_idesc_bf16_f32(kTQ, TK, 0, 0);
            const uint64_t descQ = make_smem_desc_sw128(smem_u32(sQ), 16, 1024);
            const uint64_t descK = make_smem_desc_sw128(smem_u32(sK), 16, 1024);
            uint32_t itq = 0, g = 0;
            bool ok = true;
            for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
                const int n = p.items[idx].ntiles;
                if (n == 0) continue;
                ok = mbar_wait(smem_u32(&bars.q_full), itq & 1, abortp);
                if (!ok) break;
                for (int j = 0; j < n; ++j) {
                    const uint32_t gs = g + j;
                    const int stage = gs % NS;
                    const uint32_t ph = (gs / NS) & 1, sb = gs & 1;
                    ok = mbar_wait(smem_u32(&bars.k_full[stage]), ph, abortp);
                    if (!ok) break;
                    // S[sb] was last read by the softmax of tile gs-2.  P lives in its own columns, so Q K^T could
                    // start as soon as that softmax has arrived on p_ready, but issuing it ahead of the P V of
                    // tile gs-2 delays the P V the softmax chain waits for (measured slower): keep the order
                    // P V (gs-2) -> Q K^T (gs)
                    if (gs >= 2) {
                        ok = mbar_wait(smem_u32(&bars.pv_done[sb]), ((gs >> 1) - 1) & 1, abortp);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    const uint32_t d_s = tmem + (sb ? kColS1 : kColS0);
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) {
                        const uint64_t a = descQ + (uint64_t)(((k / 4) * Q_SUB + (k % 4) * 32) >> 4);
                        const uint64_t b = descK + (uint64_t)((stage * KV_TILE + (k / 4) * KV_SUB + (k % 4) * 32) >> 4);
                        mma_ss(d_s, a, b, idesc_qk, k > 0);
                    }
                    mma_commit(smem_u32(&bars.k_empty[stage]));
                    mma_commit(smem_u32(&bars.s_full[sb]));
                    if (j == n - 1) mma_commit(smem_u32(&bars.q_empty));
                }
                g += n;
                ++itq;
            }
        }
    } else if (warp == 10) {
        // =========================== P V issuer ===========================
        if (lane == 0) {
            constexpr uint32_t idesc_pv = make_idesc_bf16_f32(kTQ, D, 0, 1);
            const uint64_t descV = make_smem_desc_sw128(smem_u32(sV), KV_SUB, 1024);
            uint32_t itq = 0, g = 0;
            bool ok = true;
            for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
                const int n = p.items[idx].ntiles;
                if (n == 0) continue;
                for (int j = 0; j < n; ++j) {
                    const uint32_t gp = g + j;
                    const int stage = gp % NS;
                    const uint32_t ph = (gp / NS) & 1, sb = gp & 1;
                    ok = mbar_wait(smem_u32(&bars.p_ready[sb]), (gp >> 1) & 1, abortp);
                    if (!ok) break;
                    ok = mbar_wait(smem_u32(&bars.v_full[stage]), ph, abortp);
                    if (!ok) break;
                    if (j == 0) {
                        ok = mbar_wait(smem_u32(&bars.o_free), (itq & 1) ^ 1, abortp);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    const uint32_t a_p = tmem + (sb ? kColP1 : kColP0);
#pragma unroll
                    for (int k = 0; k < TK / 16; ++k) {
                        const uint64_t b = descV + (uint64_t)((stage * KV_TILE + k * 2048) >> 4);
                        mma_ts(tmem + kColO, a_p + k * 8, b, idesc_pv, (j > 0 || k > 0) ? 1u : 0u);
                    }
                    mma_commit(smem_u32(&bars.v_empty[stage]));
                    mma_commit(smem_u32(&bars.pv_done[sb]));
                }
                g += n;
                ++itq;
            }
        }
    } else {
        // =========================== softmax / correction / epilogue ===========================
        const int half = warp >> 2;   // which half of the columns this thread owns
        const int tw = tid & 127;     // query row inside the tile = TMEM lane
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        uint32_t itq = 0, g = 0, xuse = 0;
        bool ok = true;
        const float c2 = p.scale_log2;
        const unsigned long long sub_mask = (p.sK >= 64) ? ~0ull : ((1ull << p.sK) - 1ull);
        // exchange one float with the partner thread of this row (bounded wait, no hardware barrier)
        auto exchange = [&](float mine, float& other) -> bool {
            const uint32_t par = xuse & 1;
            xbuf[par][half][tw] = mine;
            mbar_arrive(smem_u32(&bars.xchg));
            const bool got = mbar_wait(smem_u32(&bars.xchg), par, abortp);
            other = xbuf[par][half ^ 1][tw];
            ++xuse;
            return got;
        };
        for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
            const WorkItem it = p.items[idx];
            const int row = it.q_tile * kTQ + tw;
            const bool row_ok = row < p.N;
            if (it.ntiles == 0) {
                if (row_ok) {
                    uint4* o = reinterpret_cast<uint4*>(p.O + ((size_t)it.head * p.o_head + (size_t)row * p.o_row) + half * DC);
#pragma unroll
                    for (int c = 0; c < DC / 8; ++c) o[c] = make_uint4(0, 0, 0, 0);
                    if (half == 0) p.LSE[(size_t)it.head * p.N + row] = -INFINITY;
                }
                continue;
            }
            float m_ref = -INFINITY, l = 0.f;
            int col_next = p.tile_col[it.tile_begin];  // tile metadata is fetched one tile ahead of its use
            unsigned long long member_next = p.tile_member[it.tile_begin];
            for (int j = 0; j < it.ntiles; ++j) {
                const uint32_t gs = g + j, sb = gs & 1;
                const int kv0 = col_next * TK;
                const unsigned long long member = member_next;
                if (j + 1 < it.ntiles) {
                    col_next = p.tile_col[it.tile_begin + j + 1];
                    member_next = p.tile_member[it.tile_begin + j + 1];
                }
                const bool need_mask = (member != p.full_member) || (kv0 + TK > p.Nkv);
                const uint32_t row_bits = (uint32_t)((member >> ((tw >> p.lgBQ) * p.sK)) & sub_mask);
                const int n_valid = p.Nkv - kv0;
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.s_full[sb]), (gs >> 1) & 1, abortp));
                if (!ok) break;
                tc_fence_after();
                const uint32_t t_s = tmem + lane_base + (sb ? kColS1 : kColS0) + half * NC;
                const uint32_t t_p = tmem + lane_base + (sb ? kColP1 : kColP0) + half * (NC / 2);
                uint32_t r[NC];
#pragma unroll
                for (int c = 0; c < NC / 32; ++c) tmem_ld32(t_s + c * 32, &r[c * 32]);
                tc_wait_ld();
                if (need_mask) {
#pragma unroll
                    for (int i = 0; i < NC; ++i) {
                        const int col = half * NC + i;
                        const bool act = ((row_bits >> (col >> p.lgBKV)) & 1u) && (col < n_valid);
                        r[i] = act ? r[i] : 0xff800000u;
                    }
                }
                float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
                for (int i = 0; i < NC; i += 4) {
                    m0 = fmaxf(m0, __uint_as_float(r[i]));
                    m1 = fmaxf(m1, __uint_as_float(r[i + 1]));
                    m2 = fmaxf(m2, __uint_as_float(r[i + 2]));
                    m3 = fmaxf(m3, __uint_as_float(r[i + 3]));
                }
                float mx = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3)), mx_other;
                ok = __all_sync(0xffffffffu, exchange(mx, mx_other));
                if (!ok) break;
                const float mx2 = fmaxf(mx, mx_other) * c2;
                float alpha = 1.f;
                bool rescale = false;
                if (mx2 > m_ref + kRescaleThreshold) {
                    alpha = ex2_approx(m_ref - mx2);
                    rescale = (j > 0) && (m_ref != -INFINITY);
                    m_ref = mx2;
                }
                const float neg_m = (m_ref == -INFINITY) ? 0.f : -m_ref;
                float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
                for (int i = 0; i < NC; i += 8) {
                    float t[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) t[k] = fmaf(__uint_as_float(r[i + k]), c2, neg_m);
#pragma unroll
                    for (int k = 0; k < 8; ++k) t[k] = ex2_approx(t[k]);
                    s0 += t[0] + t[4];
                    s1 += t[1] + t[5];
                    s2 += t[2] + t[6];
                    s3 += t[3] + t[7];
#pragma unroll
                    for (int k = 0; k < 4; ++k) r[i / 2 + k] = pack_bf16x2(t[2 * k], t[2 * k + 1]);
                }
                // P[sb] was last read by the P V of tile gs-2, issued by another thread than Q K^T: make sure it is done
                if (gs >= 2) {
                    ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.pv_done[sb]), ((gs >> 1) - 1) & 1, abortp));
                    if (!ok) break;
                }
#pragma unroll
                for (int c = 0; c < NC / 32; ++c) tmem_st16(t_p + c * 16, &r[c * 16]);
                l = l * alpha + ((s0 + s1) + (s2 + s3));
                if (j > 0 && __any_sync(0xffffffffu, rescale)) {
                    const uint32_t gp = gs - 1;
                    ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.pv_done[gp & 1]), (gp >> 1) & 1, abortp));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t t_o = tmem + lane_base + kColO + half * DC;
#pragma unroll
                    for (int c = 0; c < DC / 32; ++c) {
                        uint32_t o[32];
                        tmem_ld32(t_o + c * 32, o);
                        tc_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                        tmem_st32(t_o + c * 32, o);
                    }
                }
                tc_wait_st();
                tc_fence_before();
                mbar_arrive(smem_u32(&bars.p_ready[sb]));
            }
            if (!ok) break;
            // ---- epilogue: add the two partial sums, normalise, store this thread's half of the row ----
            {
                float l_other;
                ok = __all_sync(0xffffffffu, exchange(l, l_other));
                if (!ok) break;
                const float l_tot = (half == 0) ? (l + l_other) : (l_other + l);
                const uint32_t gl = g + it.ntiles - 1;
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.pv_done[gl & 1]), (gl >> 1) & 1, abortp));
                if (!ok) break;
                tc_fence_after();
                const float inv_l = (l_tot > 0.f) ? 1.f / l_tot : 0.f;
                const float lse = (l_tot > 0.f) ? fmaf(m_ref, 0.6931471805599453f, logf(l_tot)) : -INFINITY;
                const uint32_t t_o = tmem + lane_base + kColO + half * DC;
                if (it.nparts == 1) {
                    __nv_bfloat16* orow = p.O + ((size_t)it.head * p.o_head + (size_t)row * p.o_row) + half * DC;
#pragma unroll
                    for (int c = 0; c < DC / 32; ++c) {
                        uint32_t o[32];
                        tmem_ld32(t_o + c * 32, o);
                        tc_wait_ld();
                        if (row_ok) {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                uint4 v;
                                v.x = pack_bf16x2(__uint_as_float(o[q * 8 + 0]) * inv_l, __uint_as_float(o[q * 8 + 1]) * inv_l);
                                v.y = pack_bf16x2(__uint_as_float(o[q * 8 + 2]) * inv_l, __uint_as_float(o[q * 8 + 3]) * inv_l);
                                v.z = pack_bf16x2(__uint_as_float(o[q * 8 + 4]) * inv_l, __uint_as_float(o[q * 8 + 5]) * inv_l);
                                v.w = pack_bf16x2(__uint_as_float(o[q * 8 + 6]) * inv_l, __uint_as_float(o[q * 8 + 7]) * inv_l);
                                *reinterpret_cast<uint4*>(orow + c * 32 + q * 8) = v;
                            }
                        }
                    }
                    if (row_ok && half == 0) p.LSE[(size_t)it.head * p.N + row] = lse;
                } else {
                    float* orow = p.ws_O + ((size_t)it.ws_slot * kTQ + tw) * D + half * DC;
#pragma unroll
                    for (int c = 0; c < DC / 32; ++c) {
                        uint32_t o[32];
                        tmem_ld32(t_o + c * 32, o);
                        tc_wait_ld();
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            float4 v = make_float4(__uint_as_float(o[q * 4 + 0]) * inv_l, __uint_as_float(o[q * 4 + 1]) * inv_l,
                                                   __uint_as_float(o[q * 4 + 2]) * inv_l, __uint_as_float(o[q * 4 + 3]) * inv_l);
                            *reinterpret_cast<float4*>(orow + c * 32 + q * 4) = v;
                        }
                    }
                    if (half == 0) p.ws_LSE[(size_t)it.ws_slot * kTQ + tw] = lse;
                }
                tc_fence_before();
                mbar_arrive(smem_u32(&bars.o_free));
            }
            g += it.ntiles;
            ++itq;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (tid == 0 && abort_flag) atomicExch(&p.counters->status, (int)BSA_ERR_DEVICE_TIMEOUT);
    if (warp == 9) tmem_dealloc(tmem, kTmemCols);
}

// ==========================================================================================
// Ping-pong kernel: one 128-row Q tile per CTA, TWO softmax warpgroups that take alternate KV
// tiles (warpgroup x owns the tiles whose running index has parity x, and with them S buffer x
// at d = 64 P buffer x).  While one warpgroup is in its exponential phase the other loads its scores
// and finds its row maxima, so the XU pipe and the tensor pipe both stay fed.  At d = 128 one O
// accumulator is shared: both warpgroups follow the SAME reference maximum per row, handed from tile
// to tile through shared memory (`mref`, one word per row, published right after a tile's max phase),
// and each keeps a partial row sum, converted whenever the reference it last saw has moved.  At d = 64
// each has an accumulator and a reference of its own (below).  P has its own TMEM columns, so S[x] is
// free again as soon as warpgroup x has read it into registers (`s_free`).
// A third warpgroup owns the epilogue: at the end of a work item the softmax warpgroups only hand
// over their row sums and move straight on to the next
// item's tiles; the epilogue warpgroup waits for the item's last P V, drains the accumulator,
// normalises and stores, and releases the accumulator for the next item's first P V, which cannot
// be issued before that item's first softmax tile is done anyway.
//   warps 0-3 / 4-7 : softmax warpgroups 0 / 1      warp 8 : K TMA producer   warp 11 : V TMA producer
//   warp 9 : Q K^T issuer      warp 10 : P V issuer    warps 12-15 : epilogue warpgroup (and Q tiles)
// Registers (setmaxnreg): softmax 192, epilogue 80, producers and issuers 48 per thread; the sum over the CTA,
// 256*192 + 128*80 + 128*48 = 65536, is exactly the launch allocation of 512 threads x 128.
//
// Where Q K^T reads Q, its A operand, at d = 128.  From TMEM on long lists: a 128x128x16 MMA with both operands in shared
// memory reads the full 128 B/clk for as long as it runs, so per 128-key tile 160 KB would go through shared memory (Q and
// K 64, V 32, the two TMA tiles 64) instead of 128.  The epilogue warpgroup, idle for most of a long item, moves the next
// item's Q tile from the buffer it lands in to TMEM.  With all columns taken the two warpgroups share one P buffer: tile
// j's P V has long read it when tile j+1 stores its P.  Together with the warp-uniform waits (mbar_wait_warp), builds in
// turn: 16384 tokens, 8 heads, (128,128) blocks, 19 tiles per item 177.8 -> 173.2 us.
// From shared memory on short lists, where the way through the epilogue warpgroup lies on every item's path: two Q tiles
// (the V ring gives up one of its four), loaded by the K producer.  Forward at 32768 tokens, 8 heads, n tiles per item,
// TMEM / shared memory in us: n = 1 46.8 / 41.4, 2 55.4 / 52.1, 3 68.3 / 66.0, 4 81.3 / 79.7, 6 107.6 / 106.1; at 16384
// tokens 8 67.5 / 67.5, 12 93.4 / 93.9.  Hence shared memory below eight tiles per item on average (bsa_plan::short_lists).
// Reference maximum in bf16 on long lists (kFirstRef): the maximum of the first tile that reaches a row serves the
// whole item.  bf16 and fp32 keep their relative precision over 2^100, so it does not matter how far later scores lie above
// it; from its second tile on a softmax warpgroup neither looks for maxima (64 instructions and about 300 clk per tile) nor
// takes and publishes a word per row and tile, and nothing is rescaled.  Where it fails (a row sum beyond 2^100 or undefined,
// or an output that is not finite) the epilogue marks the item, and a second pass over the marked items follows the running
// maximum as before, moved by more than 2^8 at a time.  Per 128-key tile the softmax chain falls by a fifth.  Builds in turn,
// back to back, before / after: 16384 tokens, 8 heads, (128,128) 153.5 / 144.4 us; 115200, 4 heads 1840 / 1725; 75600, 6
// heads, (64,64) 3650 / 3510, 4 heads, (32,32) 4560 / 3700.  At d = 64 (each warpgroup has its own) on lists of 32
// tiles and more: 32768 tokens, 16 heads, (256,256) 1250 / 1203; 8 heads, (32,32), 12 % independent blocks 1343 / 1284; 23296 tokens,
// 2 heads, (256,256) at 44 % 190 / 185.  The running maximum stays for half, which has no such range, and for short lists, where the second copy
// of the loop costs more than it saves (d = 128, 32768 tokens, 8 heads, two tiles per item 74 -> 82 us; d = 64, 2048 tokens, 2
// heads 16.5 -> 18.5, 10240 tokens, 8 heads, 9 tiles of runs 55 -> 63; 16384 tokens, 16 heads, (32,32), 15 tiles 244 -> 250);
// at d = 64 also for tiles of two entries ((64,64) at 48 tiles 1360 -> 1440); and for lists that are short next to the time until
// all rows of a tile have been reached (choose_list_form in bsa_api.cu has the lines).  Both forms take a row's reference from
// the same tile, so that an item whose scores do not outgrow it by 2^8 has the same bits in either.
// What the second pass costs: an item with one marked row is computed twice by its CTA.  32768 tokens, 8 heads, no item marked /
// one in a hundred / all, the running maximum in brackets: (128,128) 24 tiles 304 / 353 / 664 (329) us, (128,64) 333 / 382 / 774
// (350), (128,32) 329 / 364 / 862 (380); d = 64, 40 tiles, (128,128) 484 / 562 / 1000 (490), (128,32) 480 / 517 / 935 (475).
// Kernels and not flags in one: what an item pays at its boundary is mostly instruction fetch, and the softmax code
// has no register to spare (one kernel with both places of Q was 1-2 % slower on long lists).
//
// G: a 128-key tile is made up of G entries of the plan's tile list (T_KV = 128 / G keys each), whichever they are: the
// producers copy them one by one, and a 128-row, 128-column MMA works on a tile without gaps.  G = 1 where the logical
// key blocks have 128 keys or more.  Narrower blocks used to be Coarsened onto aligned 128-key tiles, which also compute
// their inactive neighbours, or walked in tiles of 64 keys, each with the hand-overs of a whole one.  On one GPU
// (75600 tokens, d = 128, forward, builds in turn): (64,64) blocks, 24 heads, 10 % active 17.0 -> 11.4 ms (covered over
// active pairs 1.44 both times); (32,32) 22.3 -> 14.9 ms (2.53 -> 1.92); (128,64) fp16, 12 heads, 30 % 11.7 -> 10.4 ms.
// A K tile takes G*d/64 copies (the MMA wants its rows 128 bytes x 1024 apart across entries), a V tile G (an entry's
// 64-column halves lie together, the MMA's descriptor moves from entry to entry).
//
// d = 64: two accumulators fit, so each softmax warpgroup has its own (and its own reference maximum): nothing is handed
// from tile to tile, no shared-memory round trip and vote per tile, and the epilogue adds the two up with their weights.
// Q always stays in shared memory, double-buffered (every TMEM column is taken; at d = 64 shared memory is half idle).
// Builds in turn: 3600 x 1111 tokens, 16 heads, (64,32) fp16 29.5 -> 26.4 us; 32768 tokens, 16 heads, (16,64) as 64-key
// entries 4.94 -> 4.73 ms; (256,256) 1.27 -> 1.25 ms; 2048 tokens, 2 heads 23.0 -> 22.5 us.
// TMEM columns, d = 128: S0 0, S1 128, O 256, P 384, Q 448 (or unused); d = 64: S0 0, S1 128, O0 256, O1 320, P0 384, P1 448.
// ==========================================================================================
constexpr int kPpThreads = 512;
constexpr int kPpTK = 128;  // keys of a tile

// The k-th work item of CTA b out of G: rounds of G consecutive items, alternately dealt forwards and backwards.
// Items arrive longest first, so dealing every round in the same direction would hand CTA 0 the longest item of
// every round and the last CTA the shortest; reversing every other round evens the per-CTA sums out.
__device__ __forceinline__ int cta_item_index(int k, int b, int G) { return k * G + ((k & 1) ? (G - 1 - b) : b); }

// Work item `idx` through the read-only path (items are written by the planner before the launch); past the end
// of the list the item has ntiles = -1 (an item with ntiles = 0 is a real row without active columns).
__device__ __forceinline__ WorkItem load_item(const WorkItem* items, int idx, int n_items) {
    WorkItem it;
    if (idx < n_items) {
        const int4* src = reinterpret_cast<const int4*>(items + idx);
        const int4 a = __ldg(src), b = __ldg(src + 1);
        it.head = a.x; it.q_tile = a.y; it.tile_begin = a.z; it.tile_end = a.w;
        it.part = b.x; it.nparts = b.y; it.ws_slot = b.z; it.ntiles = b.w;
    } else {
        it.head = it.q_tile = it.tile_begin = it.tile_end = it.part = it.ws_slot = 0;
        it.nparts = 1;
        it.ntiles = -1;
    }
    return it;
}

// The two fields of a work item the softmax warpgroups need, prefetched into registers with loads that stay put.
struct ItemSpan {
    int tile_begin, ntiles;  // ntiles = -1 past the end of the list
};
__device__ __forceinline__ ItemSpan load_item_span(const WorkItem* items, int idx, int n_items) {
    ItemSpan r;
    r.tile_begin = 0;
    r.ntiles = -1;
    if (idx < n_items) {
        const int* w = reinterpret_cast<const int*>(items + idx);
        r.tile_begin = ldg_pinned_s32(w + 2);
        r.ntiles = ldg_pinned_s32(w + 7);
    }
    return r;
}

// Slot and phase of a shared-memory ring, advanced once per tile (the single-thread roles sit on the path of every
// tile: no division by the ring depth there).
struct RingPos {
    int stage = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void advance(int depth) {
        if (++stage == depth) {
            stage = 0;
            phase ^= 1u;
        }
    }
};

struct __align__(8) PpBarriers {
    uint64_t q_full[2], qt_full, q_free, q_drained, o_free, o_full, e_ready, e_taken;
    uint64_t pass_done, tags_reset;
    uint64_t k_full[kMaxStages], k_empty[kMaxStages], v_full[kMaxStages], v_empty[kMaxStages];
    uint64_t s_full[2], s_free[2], p_ready[2], pv_done[2];
};

// Rounds of a CTA at most where items can be computed again: each has its own mark (an item that shared one would be computed
// again with the other, in another form).  1024 marks are what the kernel's static shared memory has left; a list of more than
// 1024 items per SM is shared out among twice as many CTAs, or more (see the launch).
constexpr int kRedoBits = 1024;
template <int V>
struct IntC {
    static constexpr int value = V;
};
// A row sum (at least 1: the reference's own weight; 0: no active block) is trusted up to 2^100.
__device__ __forceinline__ bool sum_is_doubtful(float l) { return !(l <= 1.2676506e30f); }

// Tensor-memory columns of the ping-pong kernel (Q's are in use only where Q K^T reads it from there).
template <int D>
struct PpCols {
    static constexpr bool kOwnO = (D == 64);  // an accumulator per softmax warpgroup
    static constexpr uint32_t kO0 = kColO, kO1 = kOwnO ? 320 : kColO;
    static constexpr uint32_t kP0 = kColP0, kP1 = kOwnO ? kColP1 : kColP0;
    static constexpr uint32_t kQ = 448;
};

// Tiles of a list of n entries, G entries to a tile (n <= 0: no tiles, or past the end of the list).  Where a pass leaves items
// out (n = -1, only in long forms) they count as none: the softmax warpgroups add this number up over all items, left out or not, to
// know which of them takes a tile.  Elsewhere -1 stands at the end of the list only, and either will do: zero makes long forms of half
// faster (16384 tokens, 4 heads, (64,64) 101.6 -> 99.7 us, (32,32) 144.7 -> 141.9), -1 the short ones (three short items per SM 18.0 -> 17.9).
template <int G, bool kShort>
__device__ __forceinline__ int tiles_of(int n) {
    return n > 0 ? (n + G - 1) / G : kShort ? n : 0;
}
// First keys of the entries of one tile; entries beyond the list start at N_kv, where the copy reads zeros.
template <int G, int GK>
struct TileKeys {
    int key0[G];
    __device__ __forceinline__ void load(const int32_t* cols, int e0, int end, int n_kv) {
#pragma unroll
        for (int e = 0; e < G; ++e) key0[e] = (G == 1 || e0 + e < end) ? cols[e0 + e] * GK : n_kv;
    }
};

template <int D, bool F16, int G, bool kShort, bool kFirstRef>
__global__ void __launch_bounds__(kPpThreads, 1)
bsa_attention_pp_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const AttnParams p) {
    constexpr int TK = kPpTK;
    constexpr int NSUB = D / 64;
    constexpr int Q_SUB = kTQ * 128;
    constexpr int KV_SUB = TK * 128;
    constexpr int KV_TILE = NSUB * KV_SUB;
    constexpr int GK = TK / G;  // keys of one entry of the tile list
    constexpr int GV_TILE = KV_TILE / G;
    constexpr int V_SUB = (G == 1) ? KV_SUB : GK * 128;  // a V tile holds its entries one after the other
    using Cols = PpCols<D>;
    constexpr bool kSmemQ = kShort || D == 64;  // (at d = 64 no tensor-memory columns are left for Q)
    constexpr bool kOwnO = Cols::kOwnO;
    static_assert(!(kFirstRef && (F16 || kShort)), "a row's first reference serves the whole item: long lists in bf16 only");
    static_assert(kOwnO || NSUB * Q_SUB == KV_TILE, "at d = 128 the second Q tile takes the place of a V tile");
    // dynamic shared memory starts on a 1024-byte boundary (the swizzled tiles need it); checked below
    extern __shared__ __align__(1024) uint8_t smem[];
    const int NSK = p.stages, NSV = p.stages_v - (!kOwnO && kSmemQ ? 1 : 0);
    uint8_t* sQ = smem;                                      // two Q tiles, or the landing buffer of the next one
    uint8_t* sK = sQ + (kSmemQ ? 2 : 1) * (NSUB * Q_SUB);    // NSK K tiles (a K tile lives from its load to the end of its Q K^T)
    uint8_t* sV = sK + NSK * KV_TILE;                        // NSV V tiles (a V tile lives about two tiles longer, until its P V)
    __shared__ PpBarriers bars;
    // [publishing warpgroup][row]: the reference maximum after that warpgroup's latest tile.  One 32-bit word per
    // row carries value and sequence together: reference values keep their two lowest mantissa bits clear, and
    // the word's two low bits hold (publish index + 1) mod 4, so the reader of the next tile (always the same
    // row's thread of the other warpgroup, which consumes every publish in order) needs one shared-memory
    // read, with no barrier in front of it, to know whether the value it got is the one it waits for.
    // (d = 64: each warpgroup's own reference at the end of an item, plain.  First pass under kFirstRef: [item parity][row],
    // the references as far as they are known, handed from tile to tile until every row of the warp has one; tags 0 or 1
    // from the item's first tile, by its number's second bit, then 2 and 3 in turn.)
    __shared__ uint32_t mref[2][kTQ];
    __shared__ float lfin[2][kTQ];   // [warpgroup][row]: an item's partial row sums (d = 128: in its final reference)
    __shared__ float mfin[kTQ];      // d = 128: the item's final reference maximum (log2 domain) per row
    __shared__ uint32_t redo_bits[kRedoBits / 32], redo_any;  // rounds of the CTA's items that pass 1 computes again
    __shared__ uint32_t tmem_base_s;
    __shared__ uint32_t abort_flag;


    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#ifdef BSA_TRACE
    if (tid == 0 && blockIdx.x < 4096) g_cta_times[0][blockIdx.x] = (long long)globaltimer_ns();
#endif
    if (smem_u32(smem) & 1023u) {  // never expected; fail with a status instead of corrupting tiles
        if (tid == 0) atomicExch(&p.counters->status, (int)BSA_ERR_CUDA);
        return;
    }

    if (tid == 0) {
        abort_flag = 0;
        for (int b = 0; b < 2; ++b) mbar_init(smem_u32(&bars.q_full[b]), 1);  // the Q tile has landed in shared memory
        mbar_init(smem_u32(&bars.qt_full), 128);    // epilogue threads: the Q tile is in TMEM
        mbar_init(smem_u32(&bars.q_free), 1);       // the item's last Q K^T from TMEM has completed
        mbar_init(smem_u32(&bars.q_drained), 128);  // epilogue threads: the Q tile has been read from shared memory
        mbar_init(smem_u32(&bars.o_free), 128);   // epilogue threads: accumulator drained
        mbar_init(smem_u32(&bars.o_full), 1);     // P V issuer: the item's last P V has completed
        mbar_init(smem_u32(&bars.e_ready), 256);  // softmax threads: row sums of the item are in shared memory
        mbar_init(smem_u32(&bars.e_taken), 128);  // epilogue threads: row sums read
        mbar_init(smem_u32(&bars.pass_done), 384);  // epilogue and softmax threads: the first pass is over
        mbar_init(smem_u32(&bars.tags_reset), 256);
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(smem_u32(&bars.k_full[s]), 1);
            mbar_init(smem_u32(&bars.k_empty[s]), 1);
            mbar_init(smem_u32(&bars.v_full[s]), 1);
            mbar_init(smem_u32(&bars.v_empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bars.s_full[s]), 1);
            mbar_init(smem_u32(&bars.s_free[s]), 128);
            mbar_init(smem_u32(&bars.p_ready[s]), 128);
            mbar_init(smem_u32(&bars.pv_done[s]), 1);
        }
        fence_mbar_init();
    }
    if (tid < 2 * kTQ) (&mref[0][0])[tid] = kFirstRef ? 2u : 0u;  // a tag that matches no first publish
    if (tid < kRedoBits / 32) redo_bits[tid] = 0u;
    if (tid == kTQ) redo_any = 0u;
    if (warp == 9) {
        tmem_alloc(smem_u32(&tmem_base_s), kTmemCols);
        tmem_relinquish();
    }
    if (warp == 8 && lane == 0) {
        prefetch_tensormap(&tmQ);
        prefetch_tensormap(&tmK);
        prefetch_tensormap(&tmV);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    volatile uint32_t* abortp = &abort_flag;
    // Launched with programmatic stream serialisation, this grid may start while the kernel in front of it (the task
    // organisation) is still running: everything above touches only this CTA's shared memory, TMEM and the kernel
    // parameters; nothing below runs before that kernel has completed and its writes are visible.
    grid_dependency_wait();
    const int n_items = p.counters->nitems;
    const int n_rounds = (n_items + (int)gridDim.x - 1) / (int)gridDim.x;
    // Pass 0 goes through all of the CTA's items, pass 1 (bf16) through those that the epilogue has marked.
    auto item_at = [&](auto pass_c, int kr) -> int {  // the list's index of round kr, past the end where the pass leaves it out
        if constexpr (decltype(pass_c)::value == 1) {
            const int bit = kr % kRedoBits;  // (kr runs up to two rounds past the end)
            if (!((redo_bits[bit >> 5] >> (bit & 31)) & 1u)) return n_items;
        }
        return cta_item_index(kr, blockIdx.x, gridDim.x);
    };
    // Every role between its two passes: whether there is a second one.
    auto second_pass = [&]() -> bool {
        return mbar_wait(smem_u32(&bars.pass_done), 0, abortp) && *reinterpret_cast<volatile uint32_t*>(&redo_any) != 0;
    };

    if (warp >= 12) {
        // =========================== epilogue warpgroup ===========================
        reg_dec<80>();
        const int tw = tid & 127;
        const uint32_t t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        uint32_t itn = 0;  // non-empty items seen
        uint32_t g_start = 0;  // running tile index at the start of the item
        bool ok = true;
        BSA_TRACE_DECL(tn);
        // ---- Q tiles.  d = 64: TMA into two buffers, two items ahead.  d = 128 from shared memory: the K producer loads
        // them.  From TMEM: TMA into one buffer one item ahead, then to TMEM through this warpgroup's registers. ----
        int kq = 0;       // round of the next Q tile to load
        uint32_t nq = 0;  // Q tiles loaded so far
        bool arrived = false;  // at pass_done
        auto load_q = [&](auto pass_c) {  // lane 0 of the warpgroup's first warp issues; every thread follows the item list
            WorkItem w;
            do {
                if (kq >= n_rounds) return;
                w = load_item(p.items, item_at(pass_c, kq++), n_items);
            } while (w.ntiles <= 0);
            const uint32_t b = kOwnO ? (nq & 1u) : 0u;
            if (tw == 0) {
                mbar_arrive_expect_tx(smem_u32(&bars.q_full[b]), NSUB * Q_SUB);
                tma_load_4d(smem_u32(sQ + b * NSUB * Q_SUB), &tmQ, smem_u32(&bars.q_full[b]), 0, w.q_tile * kTQ, 0, w.head);
            }
            ++nq;
        };
        uint32_t sq = 0;  // Q tiles moved to TMEM
        auto stage_q = [&](auto pass_c) -> bool {
            bool good = mbar_wait(smem_u32(&bars.q_full[0]), sq & 1, abortp);
            good = good && mbar_wait(smem_u32(&bars.q_free), (sq & 1) ^ 1, abortp);
            if (!__all_sync(0xffffffffu, good)) return false;
            tc_fence_after();
            const uint32_t t_q = tmem + ((uint32_t)((warp & 3) * 32) << 16) + Cols::kQ;
            // Swizzled 16-byte chunks of this row at a time.  Eight of them spill beside the verdict on first references; in half
            // tiles of four entries are faster with eight (16384 tokens, 4 heads, (32,32) 143.0 -> 141.1 us, 2 heads, (16,16) 172.1 -> 170.4), the
            // others are not (58594 tokens, 15 heads, (64,128) 2910 -> 3015).
            constexpr int PC = F16 && G == 4 ? 8 : 4;
#pragma unroll 1
            for (int s = 0; s < 8 * NSUB / PC; ++s) {
                uint32_t v[4 * PC];
                const uint8_t* row = sQ + (s * PC >> 3) * Q_SUB + tw * 128;
#pragma unroll
                for (int c = 0; c < PC; ++c) {
                    const uint4 w = *reinterpret_cast<const uint4*>(row + (((s * PC & 7) + c) ^ (tw & 7)) * 16);
                    v[4 * c] = w.x; v[4 * c + 1] = w.y; v[4 * c + 2] = w.z; v[4 * c + 3] = w.w;
                }
                if constexpr (PC == 8) tmem_st32(t_q + s * 32, v);
                else tmem_st16(t_q + s * 16, v);
            }
            mbar_arrive(smem_u32(&bars.q_drained));
            tc_wait_st();
            tc_fence_before();
            mbar_arrive(smem_u32(&bars.qt_full));
            if (tw == 0) good = mbar_wait(smem_u32(&bars.q_drained), sq & 1, abortp);  // then the next Q tile may land
            if (!__all_sync(0xffffffffu, good)) return false;
            ++sq;
            load_q(pass_c);
            return true;
        };
        const auto run = [&](auto pass_c) {
            constexpr int pass = decltype(pass_c)::value;
            kq = 0;
            if constexpr (kOwnO || !kSmemQ) load_q(pass_c);
            if constexpr (kOwnO) load_q(pass_c);
            WorkItem it_next = load_item(p.items, item_at(pass_c, 0), n_items);
            for (int kr = 0; kr < n_rounds && ok; ++kr) {
                const WorkItem it = it_next;
                it_next = load_item(p.items, item_at(pass_c, kr + 1), n_items);
                const int row = it.q_tile * kTQ + tw;
                const bool row_ok = row < p.N;
                if (it.ntiles < 0) continue;  // past the end of the list
                if (it.ntiles == 0) {  // no active column: zero output, LSE = -inf
                    if (row_ok && pass == 0) {
                        uint4* o = reinterpret_cast<uint4*>(p.O + ((size_t)it.head * p.o_head + (size_t)row * p.o_row));
#pragma unroll
                        for (int c = 0; c < D / 8; ++c) o[c] = make_uint4(0, 0, 0, 0);
                        p.LSE[(size_t)it.head * p.N + row] = -INFINITY;
                    }
                    continue;
                }
                // the next item's Q tile first (its Q K^T runs ahead of this item's softmax); the one TMEM buffer is
                // free after this item's last Q K^T, which comes well before its last P V
                if constexpr (!kSmemQ) {
                    while (ok && nq > sq && sq <= itn + 1) ok = stage_q(pass_c);
                    if (!ok) break;
                }
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.e_ready), itn & 1, abortp));
                if (!ok) break;
                if constexpr (kOwnO) load_q(pass_c);  // this item's scores have all been read: its buffer is free for the item after next
                // d = 64: weights of the accumulator of the item's first tile (a) and of the other one (b).  Which warpgroup took
                // the first tile follows from the tiles this CTA had before, so everything below goes by a and b and not by
                // warpgroup: an item's bits are the same wherever it stands in a CTA's list.
                const uint32_t first = g_start & 1u;
                float l_tot, m_final, wa = 1.f, wb = 1.f;
                bool doubtful = false;
                if constexpr (kOwnO) {
                    const float ma = __uint_as_float(mref[first][tw]), mb = __uint_as_float(mref[first ^ 1u][tw]);
                    m_final = fmaxf(ma, mb);
                    wa = (ma == -INFINITY) ? 0.f : ex2_approx(ma - m_final);
                    wb = (mb == -INFINITY) ? 0.f : ex2_approx(mb - m_final);
                    l_tot = fmaf(lfin[first ^ 1u][tw], wb, lfin[first][tw] * wa);
                    if (kFirstRef && pass == 0) doubtful = row_ok && (sum_is_doubtful(lfin[0][tw]) || sum_is_doubtful(lfin[1][tw]));
                } else {
                    l_tot = lfin[0][tw] + lfin[1][tw];
                    m_final = mfin[tw];
                    if (kFirstRef && pass == 0) doubtful = row_ok && sum_is_doubtful(l_tot);
                }
                mbar_arrive(smem_u32(&bars.e_taken));
                const float inv_l = (l_tot > 0.f) ? 1.f / l_tot : 0.f;
                const float lse = (l_tot > 0.f) ? fmaf(m_final, 0.6931471805599453f, logf(l_tot)) : -INFINITY;
                if (lane == 0) BSA_TRACE_POINT(11, tn, 32);
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.o_full), itn & 1, abortp));
                if (!ok) break;
                tc_fence_after();
                if (lane == 0) BSA_TRACE_POINT(11, tn, 31);
                ++itn;
                __nv_bfloat16* orow = p.O + ((size_t)it.head * p.o_head + (size_t)row * p.o_row);
                float* wrow = p.ws_O + ((size_t)it.ws_slot * kTQ + tw) * D;
                constexpr int CW = kOwnO ? 16 : 32;  // columns at a time
                const int n_tiles = tiles_of<G, kShort>(it.ntiles);  // 1: the other accumulator is stale
                g_start += (uint32_t)n_tiles;
                const float sa = inv_l * wa, sb = inv_l * wb;
                // An accumulator can overflow where the running maximum's weights of at most 2^8 would not: however small the row's
                // sum is, its outputs decide as well (d = 64: those of either accumulator, weighted by zero or not).
                uint64_t nf = pack_f32x2(0.f, 0.f);  // zero as long as every output is finite
#pragma unroll 1  // once per item: a rolled loop keeps the kernel's code small
                for (int c = 0; c < D / CW; ++c) {
                    uint32_t o[CW];
                    if constexpr (kOwnO) {
                        uint32_t ob[CW];
                        tmem_ld16(t_lane + (first ? Cols::kO1 : Cols::kO0) + c * CW, o);
                        tmem_ld16(t_lane + (first ? Cols::kO0 : Cols::kO1) + c * CW, ob);
                        tc_wait_ld();
#pragma unroll
                        for (int e = 0; e < CW; ++e) {
                            const float a = __uint_as_float(o[e]) * sa;
                            o[e] = __float_as_uint(n_tiles > 1 ? fmaf(__uint_as_float(ob[e]), sb, a) : a);
                        }
                    } else {
                        tmem_ld32(t_lane + kColO + c * CW, o);
                        tc_wait_ld();
#pragma unroll
                        for (int e = 0; e < CW; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * sa);
                    }
                    if (c == D / CW - 1) {  // the accumulator is in registers: the next item's first P V may overwrite it
                        tc_fence_before();
                        mbar_arrive(smem_u32(&bars.o_free));
                        if (lane == 0) BSA_TRACE_POINT(11, tn, 33);
                    }
                    if (kFirstRef && pass == 0) {
                        const uint64_t zero2 = pack_f32x2(0.f, 0.f);
#pragma unroll
                        for (int e = 0; e < CW; e += 2)
                            nf = fma_f32x2(pack_f32x2(__uint_as_float(o[e]), __uint_as_float(o[e + 1])), zero2, nf);
                        if (c == D / CW - 1) {
                            float f0, f1;
                            unpack_f32x2(add_f32x2(nf, zero2), f0, f1);  // (without this sum ptxas' d = 64 loops are 1.5 % slower)
                            if (__any_sync(0xffffffffu, doubtful || (row_ok && !(f0 + f1 == 0.f))) && lane == 0) {
                                atomicOr(&redo_bits[kr >> 5], 1u << (kr & 31));
                                redo_any = 1u;
                            }
                            if (kr == n_rounds - 1) {  // the verdict on the CTA's last item is in
                                mbar_arrive(smem_u32(&bars.pass_done));
                                arrived = true;
                            }
                        }
                    }
                    if (it.nparts == 1) {
                        if (row_ok) {  // 32-byte stores: every thread fills whole 32-byte sectors of its own row
#pragma unroll
                            for (int q = 0; q < CW / 16; ++q) {
                                uint32_t v[8];
#pragma unroll
                                for (int e = 0; e < 8; ++e)
                                    v[e] = pack_16x2<F16>(__uint_as_float(o[q * 16 + 2 * e]), __uint_as_float(o[q * 16 + 2 * e + 1]));
                                if constexpr (kSmemQ) {  // (long lists: the branch is the cheaper form)
                                    st_global_v8_or_2v4(orow + c * CW + q * 16, v, p.o_wide);
                                } else if (p.o_wide) {
                                    st_global_v8(orow + c * CW + q * 16, v);
                                } else {
                                    uint4* dst = reinterpret_cast<uint4*>(orow + c * CW + q * 16);
                                    dst[0] = make_uint4(v[0], v[1], v[2], v[3]);
                                    dst[1] = make_uint4(v[4], v[5], v[6], v[7]);
                                }
                            }
                        }
                    } else {  // Split-K partial: normalised fp32 rows in the workspace
#pragma unroll
                        for (int q = 0; q < CW / 8; ++q) st_global_v8(wrow + c * CW + q * 8, o + q * 8);
                    }
                }
                if (it.nparts == 1) {
                    if (row_ok) p.LSE[(size_t)it.head * p.N + row] = lse;
                } else {
                    p.ws_LSE[(size_t)it.ws_slot * kTQ + tw] = lse;
                }
                if (lane == 0) BSA_TRACE_POINT(11, tn, 34);
            }
        };
        run(IntC<0>());
        if constexpr (kFirstRef) {
            if (ok) {
                if (!arrived) mbar_arrive(smem_u32(&bars.pass_done));
                if (__all_sync(0xffffffffu, second_pass())) run(IntC<1>());
            }
        }
        if (!ok && tw == 0) {  // a Q tile in flight lands before the CTA's shared memory goes away
            const uint64_t t0 = globaltimer_ns();
            while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
        }
    } else if (warp >= 8) {
        reg_dec<48>();
        if (warp == 8 && lane == 0) {
            // =========================== K producer ===========================
            // K tiles run up to NSK tiles ahead of the Q K^T issuer and never wait for V slots (the V tiles have a
            // thread of their own in warp 11).
            // Where Q stays in shared memory at d = 128 this thread also loads it, an item's tile in front of its first K tile:
            // with two K tiles in the ring the wait for that K slot says that the last Q K^T of the item before last is done.
            uint32_t g = 0, itq = 0;
            RingPos ring;  // K ring position of tile g
            bool ok = true;
            BSA_TRACE_DECL(tn);
            const auto run = [&](auto pass_c) {
                WorkItem it_next = load_item(p.items, item_at(pass_c, 0), n_items);
                for (int kr = 0; kr < n_rounds && ok; ++kr) {
                    const WorkItem it = it_next;
                    it_next = load_item(p.items, item_at(pass_c, kr + 1), n_items);
                    if (it.ntiles <= 0) continue;
                    TileKeys<G, GK> next;
                    next.load(p.tile_col, it.tile_begin, it.tile_end, p.Nkv);
                    for (int j = it.tile_begin; j < it.tile_end; j += G, ++g, ring.advance(NSK)) {
                        const TileKeys<G, GK> cur = next;
                        if (j + G < it.tile_end) next.load(p.tile_col, j + G, it.tile_end, p.Nkv);
                        const int stage = ring.stage;
                        const uint32_t ph = ring.phase;
                        BSA_TRACE_POINT(0, tn, 19);
                        ok = mbar_wait(smem_u32(&bars.k_empty[stage]), ph ^ 1, abortp);
                        if (!ok) break;
                        BSA_TRACE_POINT(0, tn, 20);
                        if (!kOwnO && kSmemQ && j == it.tile_begin) {
                            const uint32_t b = itq++ & 1u;
                            mbar_arrive_expect_tx(smem_u32(&bars.q_full[b]), NSUB * Q_SUB);
                            tma_load_4d(smem_u32(sQ + b * NSUB * Q_SUB), &tmQ, smem_u32(&bars.q_full[b]), 0, it.q_tile * kTQ, 0, it.head);
                        }
                        mbar_arrive_expect_tx(smem_u32(&bars.k_full[stage]), KV_TILE);
                        if constexpr (G == 1) {
                            tma_load_4d(smem_u32(sK + stage * KV_TILE), &tmK, smem_u32(&bars.k_full[stage]), 0, cur.key0[0], 0, it.head);
                        } else {
#pragma unroll
                            for (int e = 0; e < G; ++e)
#pragma unroll
                                for (int s = 0; s < NSUB; ++s)
                                    tma_load_4d(smem_u32(sK + stage * KV_TILE + s * KV_SUB + e * GK * 128), &tmK,
                                                smem_u32(&bars.k_full[stage]), 0, cur.key0[e], s, it.head);
                        }
                        BSA_TRACE_POINT(0, tn, 21);
                    }
                }
            };
            run(IntC<0>());
            if constexpr (kFirstRef) if (ok && second_pass()) run(IntC<1>());
            if (!ok) {
                const uint64_t t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
            }
        } else if (warp == 11 && lane == 0) {
            // =========================== V producer ===========================
            uint32_t g = 0;
            RingPos ring;  // V ring position of tile g
            bool ok = true;
            const bool withhold = *reinterpret_cast<volatile int*>(&g_withhold_arrival) != 0;  // test hook, see above
            const auto run = [&](auto pass_c) {
                WorkItem it_next = load_item(p.items, item_at(pass_c, 0), n_items);
                for (int kr = 0; kr < n_rounds && ok; ++kr) {
                    const WorkItem it = it_next;
                    it_next = load_item(p.items, item_at(pass_c, kr + 1), n_items);
                    if (it.ntiles <= 0) continue;
                    TileKeys<G, GK> next;
                    next.load(p.tile_col, it.tile_begin, it.tile_end, p.Nkv);
                    for (int j = it.tile_begin; j < it.tile_end; j += G, ++g, ring.advance(NSV)) {
                        const TileKeys<G, GK> cur = next;
                        if (j + G < it.tile_end) next.load(p.tile_col, j + G, it.tile_end, p.Nkv);
                        const int stage = ring.stage;
                        const uint32_t ph = ring.phase;
                        if (withhold && g == 0) continue;  // this tile never arrives
                        ok = mbar_wait(smem_u32(&bars.v_empty[stage]), ph ^ 1, abortp);
                        if (!ok) break;
                        mbar_arrive_expect_tx(smem_u32(&bars.v_full[stage]), KV_TILE);
#pragma unroll
                        for (int e = 0; e < G; ++e)
                            tma_load_4d(smem_u32(sV + stage * KV_TILE + e * GV_TILE), &tmV, smem_u32(&bars.v_full[stage]), 0,
                                        cur.key0[e], 0, it.head);
                    }
                }
            };
            run(IntC<0>());
            if constexpr (kFirstRef) if (ok && second_pass()) run(IntC<1>());
            if (!ok) {
                const uint64_t t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
            }
        } else if (warp == 9 && lane == 0) {
            // =========================== Q K^T issuer ===========================
            constexpr uint32_t idesc_qk = make_idesc_f32(kTQ, TK, 0, 0, F16);
            const uint64_t descQ0 = make_smem_desc_sw128(smem_u32(sQ), 16, 1024);
            const uint64_t descK = make_smem_desc_sw128(smem_u32(sK), 16, 1024);
            RingPos ring;  // K ring position of the tile being issued
            uint32_t itq = 0, g = 0;
            bool ok = true;
            BSA_TRACE_DECL(tn);
            BSA_PH_DECL;
            const auto run = [&](auto pass_c) {
                int n_next = tiles_of<G, kShort>(load_item(p.items, item_at(pass_c, 0), n_items).ntiles);
                for (int kr = 0; kr < n_rounds && ok; ++kr) {
                    const int n = n_next;
                    n_next = tiles_of<G, kShort>(load_item(p.items, item_at(pass_c, kr + 1), n_items).ntiles);
                    if (n <= 0) continue;
                    const uint32_t qb = kSmemQ ? (itq & 1u) : 0u;  // this item's Q buffer
                    ok = kSmemQ ? mbar_wait(smem_u32(&bars.q_full[qb]), (itq >> 1) & 1, abortp)
                                : mbar_wait(smem_u32(&bars.qt_full), itq & 1, abortp);
                    if (!ok) break;
                    const uint64_t descQ = descQ0 + (uint64_t)((qb * NSUB * Q_SUB) >> 4);
                    for (int j = 0; j < n; ++j, ring.advance(NSK)) {
                        const uint32_t gs = g + j;
                        const int stage = ring.stage;
                        const uint32_t ph = ring.phase, sb = gs & 1;
                        // K tile present, and S[sb] read into registers by the softmax of tile gs-2
                        if (gs >= 2)
                            ok = mbar_wait2(smem_u32(&bars.s_free[sb]), ((gs >> 1) - 1) & 1, smem_u32(&bars.k_full[stage]), ph, abortp);
                        else
                            ok = mbar_wait(smem_u32(&bars.k_full[stage]), ph, abortp);
                        if (!ok) break;
                        BSA_PH(0);
                        BSA_STAMP(0, gs, 0);
                        BSA_TRACE_POINT(1, tn, 6);
                        tc_fence_after();
                        const uint32_t d_s = tmem + (sb ? kColS1 : kColS0);
#pragma unroll(kSmemQ ? 4 : 8)  // (all eight with both operands' descriptors do not fit this thread's registers)
                        for (int k = 0; k < D / 16; ++k) {
                            const uint64_t b = descK + (uint64_t)((stage * KV_TILE + (k / 4) * KV_SUB + (k % 4) * 32) >> 4);
                            if constexpr (kSmemQ)
                                mma_ss(d_s, descQ + (uint64_t)(((k / 4) * Q_SUB + (k % 4) * 32) >> 4), b, idesc_qk, k > 0);
                            else
                                mma_ts(d_s, tmem + Cols::kQ + k * 8, b, idesc_qk, k > 0);
                        }
                        mma_commit(smem_u32(&bars.k_empty[stage]));
                        mma_commit(smem_u32(&bars.s_full[sb]));
                        BSA_PH(1);
                        BSA_STAMP(0, gs, 1);
#ifdef BSA_PHASES
                        ++ph_n;
#endif
                        BSA_TRACE_POINT(1, tn, 2);
                        if (!kSmemQ && j == n - 1) mma_commit(smem_u32(&bars.q_free));
                    }
                    g += n;
                    ++itq;
                }
            };
            run(IntC<0>());
            if constexpr (kFirstRef) if (ok && second_pass()) run(IntC<1>());
#ifdef BSA_PHASES
            if (blockIdx.x == 1) { g_trace[0][0] = ph_acc[0]; g_trace[0][1] = ph_acc[1]; g_trace[0][8] = ph_n; }
#endif
        } else if (warp == 10 && lane == 0) {
            // =========================== P V issuer ===========================
            constexpr uint32_t idesc_pv = make_idesc_f32(kTQ, D, 0, 1, F16);
            const uint64_t descV = make_smem_desc_sw128(smem_u32(sV), V_SUB, 1024);
            RingPos ring;  // V ring position of the tile being issued
            uint32_t itq = 0, g = 0;
            bool ok = true;
            BSA_TRACE_DECL(tn);
            BSA_PH_DECL;
            const auto run = [&](auto pass_c) {
                int n_next = tiles_of<G, kShort>(load_item(p.items, item_at(pass_c, 0), n_items).ntiles);
                for (int kr = 0; kr < n_rounds && ok; ++kr) {
                    const int n = n_next;
                    n_next = tiles_of<G, kShort>(load_item(p.items, item_at(pass_c, kr + 1), n_items).ntiles);
                    if (n <= 0) continue;
                    for (int j = 0; j < n; ++j, ring.advance(NSV)) {
                        const uint32_t gp = g + j;
                        const int stage = ring.stage;
                        const uint32_t ph = ring.phase, sb = gp & 1;
                        // V tile present (normally long before), accumulator drained by the epilogue (first tile of an
                        // item), and last the P tile, which is the one this thread normally waits for
                        if (j == 0) {
                            ok = mbar_wait(smem_u32(&bars.o_free), (itq & 1) ^ 1, abortp);
                            if (!ok) break;
                        }
                        ok = mbar_wait2(smem_u32(&bars.v_full[stage]), ph, smem_u32(&bars.p_ready[sb]), (gp >> 1) & 1, abortp);
                        if (!ok) break;
                        BSA_PH(0);
                        BSA_STAMP(1, gp, 0);
                        BSA_TRACE_POINT(10, tn, 3);

                        tc_fence_after();
                        const uint32_t a_p = tmem + (sb ? Cols::kP1 : Cols::kP0), d_o = tmem + (sb ? Cols::kO1 : Cols::kO0);
#pragma unroll
                        for (int k = 0; k < TK / 16; ++k) {
                            const uint64_t b = descV + (uint64_t)((stage * KV_TILE + (k / (GK / 16)) * GV_TILE + (k % (GK / 16)) * 2048) >> 4);
                            mma_ts(d_o, a_p + k * 8, b, idesc_pv, (j > (kOwnO ? 1 : 0) || k > 0) ? 1u : 0u);
                        }
                        mma_commit(smem_u32(&bars.v_empty[stage]));
                        mma_commit(smem_u32(&bars.pv_done[sb]));
                        if (j == n - 1) mma_commit(smem_u32(&bars.o_full));
                        BSA_PH(1);
                        BSA_STAMP(1, gp, 1);
#ifdef BSA_PHASES
                        ++ph_n;
#endif
                        BSA_TRACE_POINT(10, tn, 5);
                    }
                    g += n;
                    ++itq;
                }
            };
            run(IntC<0>());
            if constexpr (kFirstRef) if (ok && second_pass()) run(IntC<1>());
#ifdef BSA_PHASES
            if (blockIdx.x == 1) { g_trace[1][0] = ph_acc[0]; g_trace[1][1] = ph_acc[1]; g_trace[1][8] = ph_n; }
#endif
        }
    } else {
        // =========================== softmax warpgroup x ===========================
        reg_inc<192>();
        const int x = warp >> 2;
        const int tw = tid & 127;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t t_s = tmem + lane_base + (x ? kColS1 : kColS0);
        const uint32_t t_p = tmem + lane_base + (x ? Cols::kP1 : Cols::kP0);
        const uint32_t t_o = tmem + lane_base + (x ? Cols::kO1 : Cols::kO0);
        uint32_t g = 0;          // running tile index at the start of the current item (all warpgroups agree)
        uint32_t itn = 0;        // non-empty items finished
        uint32_t g0 = 0;         // running tile index at the start of this pass
        bool ok = true;
        BSA_TRACE_DECL(tn);
        const float c2 = p.scale_log2;
        // Membership (64-row, 128-key blocks, 75600 tokens, 12 heads: 5.74 -> 5.27 ms against reading the 64-bit word and
        // the column of every tile in every thread): each half-warp of 16 rows lies inside one logical row block, and a
        // tile has at most eight key sub-blocks, so lane l of a half-warp fetches the bit of sub-block l for the
        // half-warp's rows and one ballot hands all of them to every lane.  Plans whose entries have a single membership
        // bit need no loads at all.
        const int nb = G * p.sK, l16 = lane & 15;
        const bool has_bits = p.full_member != 1ull;
        const int mbit = (((tw & ~15) >> p.lgBQ) * p.sK) + (l16 & (p.sK - 1));
        const int ment = l16 >> p.lgSK;  // entry of the tile this lane's bit belongs to
        const uint32_t full_bits = (1u << nb) - 1u, full_ballot = full_bits | (full_bits << 16);
        const int32_t* mwords = reinterpret_cast<const int32_t*>(p.tile_member) + (mbit >> 5);
        auto load_bit = [&](int entry, int end) -> uint32_t {  // word that holds this lane's bit (0 beyond the list)
            if (l16 >= nb || entry + ment >= end) return 0u;
            return has_bits ? (uint32_t)ldg_pinned_s32(mwords + 2 * (int64_t)(entry + ment)) : 0xffffffffu;
        };
        BSA_PH_DECL;
        // The reference after global tile t (taken by the other warpgroup), given a word read earlier from its slot:
        // if that word already carries the publish's tag it is used, else the slot is polled (bounded).
        auto take_reference = [&](uint32_t t, uint32_t word, float& m_out) -> bool {
            const uint32_t tag = ((t >> 1) - (g0 >> 1) + 1) & 3u;
            if ((word & 3u) != tag) {
                volatile uint32_t* slot = &mref[x ^ 1][tw];
                long long t0 = 0;
                uint32_t spins = 0;
                while (true) {
                    word = *slot;
                    if ((word & 3u) == tag) break;
                    if ((++spins & 63u) == 0) {
                        if (*abortp) return false;
                        const long long now = clock64();
                        if (t0 == 0) t0 = now;
                        if (now - t0 > *reinterpret_cast<volatile long long*>(&g_wait_limit_cycles)) {
                            *abortp = 1;
                            return false;
                        }
                    }
                }
            }
            m_out = __uint_as_float(word & ~3u);
            return true;
        };
        // polls a reference's word until it carries the tag (bounded)
        auto take_word = [&](volatile uint32_t* slot, uint32_t tag, float& m_out) -> bool {
            uint32_t word = *slot;
            long long t0 = 0;
            for (uint32_t spins = 1; (word & 3u) != tag; ++spins) {
                if ((spins & 63u) == 0) {
                    if (*abortp) return false;
                    const long long now = clock64();
                    if (t0 == 0) t0 = now;
                    if (now - t0 > *reinterpret_cast<volatile long long*>(&g_wait_limit_cycles)) {
                        *abortp = 1;
                        return false;
                    }
                }
                word = *slot;
            }
            m_out = __uint_as_float(word & ~3u);
            return true;
        };
        bool again = true;
        if constexpr (kFirstRef) {
            // work items are fetched two items ahead and the first tile's metadata one item ahead, so that neither the
            // item nor the metadata that depends on it is waited for at an item boundary
            ItemSpan it_next = load_item_span(p.items, item_at(IntC<0>(), 0), n_items);
            ItemSpan it_next2 = load_item_span(p.items, item_at(IntC<0>(), 1), n_items);
            int last_col = 0;
            uint32_t first_word = 0;
            {
                const int j0n = ((g & 1) == (uint32_t)x) ? 0 : 1;
                first_word = load_bit(it_next.tile_begin + j0n * G, it_next.tile_begin + it_next.ntiles);
                if (it_next.ntiles > 0) last_col = ldg_pinned_s32(p.tile_col + it_next.tile_begin + it_next.ntiles - 1);
            }
            for (int kr = 0; kr < n_rounds && ok; ++kr) {
                const ItemSpan it = it_next;
                it_next = it_next2;
                it_next2 = load_item_span(p.items, item_at(IntC<0>(), kr + 2), n_items);
                const int n = tiles_of<G, kShort>(it.ntiles), end = it.tile_begin + it.ntiles;
                uint32_t word_next = first_word;
                // keys of the last tile that exist (columns are ascending, so only its last entry can be ragged)
                const int n_valid = ((it.ntiles - 1) & (G - 1)) * GK + (p.Nkv - last_col * GK);
                {   // the next item's first tile of this warpgroup: its parity follows from g + n
                    const int j0n = (((g + n) & 1) == (uint32_t)x) ? 0 : 1;
                    first_word = load_bit(it_next.tile_begin + j0n * G, it_next.tile_begin + it_next.ntiles);
                    if (it_next.ntiles > 0) last_col = ldg_pinned_s32(p.tile_col + it_next.tile_begin + it_next.ntiles - 1);
                }
                if (n <= 0) continue;  // the epilogue warpgroup writes the empty rows
                float m_ref = -INFINITY, l = 0.f;
                bool settled = false;  // every row of the warp has its reference
                // first local tile index of this warpgroup inside the item
                const int j0 = ((g & 1) == (uint32_t)x) ? 0 : 1;
                for (int j = j0; j < n; j += 2) {
                    const uint32_t gs = g + j;
                    uint32_t ballot = full_ballot;
                    if (G > 1 || has_bits) {
                        ballot = __ballot_sync(0xffffffffu, (word_next >> (mbit & 31)) & 1u);
                        if (j + 2 < n) word_next = load_bit(it.tile_begin + (j + 2) * G, end);
                    }
                    const bool need_mask = ballot != full_ballot;
                    const uint32_t row_bits = (ballot >> (lane & 16)) & full_bits;
                    const bool ragged = (j == n - 1) && n_valid < TK;
                    if (lane == 0 && j == j0) BSA_TRACE_POINT(2 + warp, tn, 35);
                    BSA_PH(7);
                    ok = mbar_wait_warp(smem_u32(&bars.s_full[x]), (gs >> 1) & 1, abortp);
                    if (!ok) break;
                    BSA_PH(0);
                    if (lane == 0) BSA_STAMP(2 + warp, gs, 0);
                    if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 10);
                    tc_fence_after();
                    uint32_t r[TK];
#pragma unroll
                    for (int c = 0; c < TK / 32; ++c) tmem_ld32(t_s + c * 32, &r[c * 32]);
                    tc_wait_ld();
                    BSA_PH(1);
                    tc_fence_before();
                    mbar_arrive(smem_u32(&bars.s_free[x]));  // S[x] is in registers: the next Q K^T into it may start
                    if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 11);
                    if (need_mask) {
                        // a sub-block has at least 16 key columns: one activity bit per 16, one instruction per element
                        // (skipping the exponentials of 32 columns that no row of the warp needs brought nothing)
#pragma unroll
                        for (int gq = 0; gq < TK / 16; ++gq) {
                            const bool grp = (row_bits >> ((gq * 16) >> p.lgBKV)) & 1u;
#pragma unroll
                            for (int i = gq * 16; i < gq * 16 + 16; ++i) r[i] = grp ? r[i] : 0xff800000u;
                        }
                    }
                    if (ragged) {
#pragma unroll
                        for (int i = 0; i < TK; ++i) r[i] = (i < n_valid) ? r[i] : 0xff800000u;
                    }
                    if (!settled) {  // the item's first tile, and where some row has not been reached yet
                        float m_prev = -INFINITY;
                        if (kOwnO) m_prev = m_ref;
                        else if (j > 0) {  // (published, since this warp is not settled; its slot is not written again before this tile's P V)
                            ok = __all_sync(0xffffffffu, take_word(&mref[itn & 1][tw], (j == 1) ? (itn >> 1) & 1u : 2u + (j & 1u), m_prev));
                            if (!ok) break;
                        }
                        if (!__all_sync(0xffffffffu, m_prev != -INFINITY)) {
                            float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
                            for (int i = 0; i < TK; i += 8) {
                                m0 = max3(m0, __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
                                m1 = max3(m1, __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3]));
                                m2 = max3(m2, __uint_as_float(r[i + 4]), __uint_as_float(r[i + 5]));
                                m3 = max3(m3, __uint_as_float(r[i + 6]), __uint_as_float(r[i + 7]));
                            }
                            const float mx2 = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3)) * c2;
                            if (m_prev == -INFINITY) m_prev = kOwnO ? mx2 : __uint_as_float(__float_as_uint(mx2) & ~3u);  // two low bits clear (see mref)
                            if (!kOwnO) *reinterpret_cast<volatile uint32_t*>(&mref[itn & 1][tw]) =
                                __float_as_uint(m_prev) | ((j == 0) ? (itn >> 1) & 1u : 3u - (j & 1u));
                        }
                        m_ref = m_prev;
                        settled = __all_sync(0xffffffffu, m_ref != -INFINITY);
                    }
                    const float neg_m = (m_ref == -INFINITY) ? 0.f : -m_ref;
                    const uint64_t c22 = pack_f32x2(c2, c2), nm2 = pack_f32x2(neg_m, neg_m);
                    uint64_t sum01 = pack_f32x2(0.f, 0.f), sum23 = sum01;
                    // P[x] was last read by the P V of tile gs-2 (normally long complete).  With d = 64 it is waited for
                    // here and the P tile stored 32 columns at a time while the next columns are still being exponentiated
                    // (+4 % on Stress-B); with d = 128 the stores follow the loop (the split loop was 1-2 % slower there).
                    constexpr bool kStoreInLoop = (D == 64);
                    if (kStoreInLoop && gs >= 2) {
                        ok = mbar_wait_warp(smem_u32(&bars.pv_done[x]), ((gs >> 1) - 1) & 1, abortp);
                        if (!ok) break;
                        tc_fence_after();
                    }
#pragma unroll
                    for (int i = 0; i < TK; i += 4) {
                        float x0, x1, x2, x3;
                        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), c22, nm2), x0, x1);
                        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(r[i + 2]), __uint_as_float(r[i + 3])), c22, nm2), x2, x3);
                        const float p0 = ex2_approx(x0), p1 = ex2_approx(x1), p2 = ex2_approx(x2), p3 = ex2_approx(x3);
                        sum01 = add_f32x2(sum01, pack_f32x2(p0, p1));
                        sum23 = add_f32x2(sum23, pack_f32x2(p2, p3));
                        r[i / 2] = pack_16x2<F16>(p0, p1);
                        r[i / 2 + 1] = pack_16x2<F16>(p2, p3);
                        if (kStoreInLoop && (i & 31) == 28) tmem_st16(t_p + (i >> 5) * 16, &r[(i >> 5) * 16]);
                    }
                    float s0, s1, s2, s3;
                    unpack_f32x2(sum01, s0, s1);
                    unpack_f32x2(sum23, s2, s3);
                    l += (s0 + s1) + (s2 + s3);
#ifdef BSA_PHASES
                    {
                        float f0_ = l;
                        uint32_t u0_ = r[TK / 2 - 1];
                        asm volatile("mov.b32 %0, %0;\n\tmov.b32 %1, %1;" : "+f"(f0_), "+r"(u0_));
                    }
#endif
                    BSA_PH(4);
                    if (lane == 0) BSA_STAMP(2 + warp, gs, 1);
                    if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 14);
                    if (!kStoreInLoop) {
                        if (gs >= 1) {  // the P tile before this one (other warpgroup's) must have been consumed
                            ok = mbar_wait_warp(smem_u32(&bars.pv_done[x ^ 1]), ((gs - 1) >> 1) & 1, abortp);
                            if (!ok) break;
                            tc_fence_after();
                        }
                        BSA_PH(5);
                        if (lane == 0) BSA_STAMP(2 + warp, gs, 2);
#pragma unroll
                        for (int c = 0; c < TK / 32; ++c) tmem_st16(t_p + c * 16, &r[c * 16]);
                    }
                    tc_wait_st();
                    tc_fence_before();
                    mbar_arrive(smem_u32(&bars.p_ready[x]));
                    BSA_PH(6);
                    if (lane == 0) BSA_STAMP(2 + warp, gs, 3);
#ifdef BSA_PHASES
                    ++ph_n;
#endif
                    if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 16);
                }
                if (!ok) break;
                // ---- hand this warpgroup's row sums to the epilogue warpgroup ----
                {
                    // the previous item's sums must have been read
                    ok = mbar_wait_warp(smem_u32(&bars.e_taken), (itn & 1) ^ 1, abortp);
                    if (!ok) break;
                    lfin[x][tw] = l;
                    if (kOwnO) mref[x][tw] = __float_as_uint(m_ref);
                    else if (((g + n - 1) & 1) == (uint32_t)x) mfin[tw] = m_ref;  // whoever took the last tile knows the reference of every row
                    mbar_arrive(smem_u32(&bars.e_ready));
                    ++itn;
                    if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 30);
                }
                g += n;
                BSA_PH(7);  // item boundary: sums handed over, next item's first tile not yet waited for
            }
            // ---- pass 1: the items whose first reference did not serve, with a reference that follows the running maximum ----
            if (ok) {
                mbar_arrive(smem_u32(&bars.pass_done));
                again = __all_sync(0xffffffffu, second_pass());
                if (!kOwnO && again) {  // everything has been read: the tags start over
                    mref[x][tw] = 0u;
                    mbar_arrive(smem_u32(&bars.tags_reset));
                    again = ok = mbar_wait_warp(smem_u32(&bars.tags_reset), 0, abortp);
                }
            }
        }
        g0 = g;
        if (ok && again) {
            // work items are fetched two items ahead and the first tile's metadata one item ahead, so that neither the
            // item nor the metadata that depends on it is waited for at an item boundary
            ItemSpan it_next = load_item_span(p.items, item_at(IntC<kFirstRef ? 1 : 0>(), 0), n_items);
            ItemSpan it_next2 = load_item_span(p.items, item_at(IntC<kFirstRef ? 1 : 0>(), 1), n_items);
            int last_col = 0;
            uint32_t first_word = 0;
            {
                const int j0n = ((g & 1) == (uint32_t)x) ? 0 : 1;
                first_word = load_bit(it_next.tile_begin + j0n * G, it_next.tile_begin + it_next.ntiles);
                if (it_next.ntiles > 0) last_col = ldg_pinned_s32(p.tile_col + it_next.tile_begin + it_next.ntiles - 1);
            }
            for (int kr = 0; kr < n_rounds && ok; ++kr) {
                const ItemSpan it = it_next;
                it_next = it_next2;
                it_next2 = load_item_span(p.items, item_at(IntC<kFirstRef ? 1 : 0>(), kr + 2), n_items);
                const int n = tiles_of<G, kShort>(it.ntiles), end = it.tile_begin + it.ntiles;
                uint32_t word_next = first_word;
                // keys of the last tile that exist (columns are ascending, so only its last entry can be ragged)
                const int n_valid = ((it.ntiles - 1) & (G - 1)) * GK + (p.Nkv - last_col * GK);
                {   // the next item's first tile of this warpgroup: its parity follows from g + n
                    const int j0n = (((g + n) & 1) == (uint32_t)x) ? 0 : 1;
                    first_word = load_bit(it_next.tile_begin + j0n * G, it_next.tile_begin + it_next.ntiles);
                    if (it_next.ntiles > 0) last_col = ldg_pinned_s32(p.tile_col + it_next.tile_begin + it_next.ntiles - 1);
                }
                if (n <= 0) continue;  // the epilogue warpgroup writes the empty rows
                float m_know = -INFINITY;  // reference maximum this thread's partial sum l is expressed in
                float l = 0.f;
                // first local tile index of this warpgroup inside the item
                const int j0 = ((g & 1) == (uint32_t)x) ? 0 : 1;
                for (int j = j0; j < n; j += 2) {
                    const uint32_t gs = g + j;
                    uint32_t ballot = full_ballot;
                    if (G > 1 || has_bits) {
                        ballot = __ballot_sync(0xffffffffu, (word_next >> (mbit & 31)) & 1u);
                        if (j + 2 < n) word_next = load_bit(it.tile_begin + (j + 2) * G, end);
                    }
                    const bool need_mask = ballot != full_ballot;
                    const uint32_t row_bits = (ballot >> (lane & 16)) & full_bits;
                    const bool ragged = (j == n - 1) && n_valid < TK;
                    if (lane == 0 && j == j0) BSA_TRACE_POINT(2 + warp, tn, 35);
                    BSA_PH(7);
                    ok = mbar_wait_warp(smem_u32(&bars.s_full[x]), (gs >> 1) & 1, abortp);
                    if (!ok) break;
                    BSA_PH(0);
                    if (lane == 0) BSA_STAMP(2 + warp, gs, 0);
                    if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 10);
                    tc_fence_after();
                    uint32_t r[TK];
#pragma unroll
                    for (int c = 0; c < TK / 32; ++c) tmem_ld32(t_s + c * 32, &r[c * 32]);
                    tc_wait_ld();
                    BSA_PH(1);
                    tc_fence_before();
                    mbar_arrive(smem_u32(&bars.s_free[x]));  // S[x] is in registers: the next Q K^T into it may start
                    if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 11);
                    // The previous tile's reference has normally been published by now: its slot is read here and the
                    // word checked after the max phase, so that the shared-memory round trip overlaps that phase.
                    uint32_t ref_word = 0;
                    if constexpr (!kOwnO) ref_word = *reinterpret_cast<volatile uint32_t*>(&mref[x ^ 1][tw]);
                    if (need_mask) {
                        // a sub-block has at least 16 key columns: one activity bit per 16, one instruction per element
                        // (skipping the exponentials of 32 columns that no row of the warp needs brought nothing)
#pragma unroll
                        for (int gq = 0; gq < TK / 16; ++gq) {
                            const bool grp = (row_bits >> ((gq * 16) >> p.lgBKV)) & 1u;
#pragma unroll
                            for (int i = gq * 16; i < gq * 16 + 16; ++i) r[i] = grp ? r[i] : 0xff800000u;
                        }
                    }
                    if (ragged) {
#pragma unroll
                        for (int i = 0; i < TK; ++i) r[i] = (i < n_valid) ? r[i] : 0xff800000u;
                    }
                    float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
                    for (int i = 0; i < TK; i += 8) {
                        m0 = max3(m0, __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
                        m1 = max3(m1, __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3]));
                        m2 = max3(m2, __uint_as_float(r[i + 4]), __uint_as_float(r[i + 5]));
                        m3 = max3(m3, __uint_as_float(r[i + 6]), __uint_as_float(r[i + 7]));
                    }
                    const float mx2 = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3)) * c2;
#ifdef BSA_TRACE
                    if (lane == 0 && mx2 != 12345.f) BSA_TRACE_POINT(2 + warp, tn, 17);
#endif
                    if constexpr (!kOwnO) {
                        // ---- reference maximum handed over from the previous tile (other warpgroup) ----
                        float m_prev = -INFINITY;
                        if (gs > g0) {  // every publish is consumed, in order, also across item boundaries (the tags rely on it)
                            float m_taken;
                            if (__all_sync(0xffffffffu, (ref_word & 3u) == ((((gs - 1) >> 1) - (g0 >> 1) + 1) & 3u))) {
                                m_taken = __uint_as_float(ref_word & ~3u);
                            } else {
                                ok = __all_sync(0xffffffffu, take_reference(gs - 1, ref_word, m_taken));
                                if (!ok) break;
                            }
                            if (j > 0) m_prev = m_taken;  // the previous tile belongs to this item
                        }
#ifdef BSA_PHASES
                        {
                            float f0_ = mx2, f1_ = m_prev;  // real instructions that read the values: the clock is read after them
                            asm volatile("mov.b32 %0, %0;\n\tmov.b32 %1, %1;" : "+f"(f0_), "+f"(f1_));
                        }
#endif
                        BSA_PH(2);
#ifdef BSA_TRACE
                        if (lane == 0 && m_prev != 12345.f) BSA_TRACE_POINT(2 + warp, tn, 18);
#endif
                        if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 12);
                        if (m_prev != m_know) {  // the other warpgroup moved the reference since this thread last looked
                            l *= ex2_approx(m_know - m_prev);  // m_know = -inf only while l = 0
                            m_know = m_prev;
                        }
                    }
                    float alpha = 1.f;
                    bool rescale = false;
                    if (mx2 > m_know + kRescaleThreshold) {
                        const float m_new = kOwnO ? mx2 : __uint_as_float(__float_as_uint(mx2) & ~3u);  // two low bits clear (see mref)
                        alpha = ex2_approx(m_know - m_new);
                        rescale = (j > (kOwnO ? 1 : 0)) && (m_know != -INFINITY);
                        l *= alpha;
                        m_know = m_new;
                    }
                    if constexpr (!kOwnO) {
                        // publish: the next tile's warpgroup may take its decision
                        *reinterpret_cast<volatile uint32_t*>(&mref[x][tw]) = __float_as_uint(m_know) | (((gs >> 1) - (g0 >> 1) + 1) & 3u);
                    }
                    BSA_PH(3);
                    const float neg_m = (m_know == -INFINITY) ? 0.f : -m_know;
                    const uint64_t c22 = pack_f32x2(c2, c2), nm2 = pack_f32x2(neg_m, neg_m);
                    uint64_t sum01 = pack_f32x2(0.f, 0.f), sum23 = sum01;
                    // P[x] was last read by the P V of tile gs-2 (normally long complete).  With d = 64 it is waited for
                    // here and the P tile stored 32 columns at a time while the next columns are still being exponentiated
                    // (+4 % on Stress-B); with d = 128 the stores follow the loop (the split loop was 1-2 % slower there).
                    constexpr bool kStoreInLoop = (D == 64);
                    if (kStoreInLoop && gs >= 2) {
                        ok = mbar_wait_warp(smem_u32(&bars.pv_done[x]), ((gs >> 1) - 1) & 1, abortp);
                        if (!ok) break;
                        tc_fence_after();
                    }
#pragma unroll
                    for (int i = 0; i < TK; i += 4) {
                        float x0, x1, x2, x3;
                        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), c22, nm2), x0, x1);
                        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(r[i + 2]), __uint_as_float(r[i + 3])), c22, nm2), x2, x3);
                        const float p0 = ex2_approx(x0), p1 = ex2_approx(x1), p2 = ex2_approx(x2), p3 = ex2_approx(x3);
                        sum01 = add_f32x2(sum01, pack_f32x2(p0, p1));
                        sum23 = add_f32x2(sum23, pack_f32x2(p2, p3));
                        r[i / 2] = pack_16x2<F16>(p0, p1);
                        r[i / 2 + 1] = pack_16x2<F16>(p2, p3);
                        if (kStoreInLoop && (i & 31) == 28) tmem_st16(t_p + (i >> 5) * 16, &r[(i >> 5) * 16]);
                    }
                    float s0, s1, s2, s3;
                    unpack_f32x2(sum01, s0, s1);
                    unpack_f32x2(sum23, s2, s3);
                    l += (s0 + s1) + (s2 + s3);
#ifdef BSA_PHASES
                    {
                        float f0_ = l;
                        uint32_t u0_ = r[TK / 2 - 1];
                        asm volatile("mov.b32 %0, %0;\n\tmov.b32 %1, %1;" : "+f"(f0_), "+r"(u0_));
                    }
#endif
                    BSA_PH(4);
                    if (lane == 0) BSA_STAMP(2 + warp, gs, 1);
                    if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 14);
                    if (!kStoreInLoop) {
                        if (gs >= 1) {  // the P tile before this one (other warpgroup's) must have been consumed
                            ok = mbar_wait_warp(smem_u32(&bars.pv_done[x ^ 1]), ((gs - 1) >> 1) & 1, abortp);
                            if (!ok) break;
                            tc_fence_after();
                        }
                        BSA_PH(5);
                        if (lane == 0) BSA_STAMP(2 + warp, gs, 2);
#pragma unroll
                        for (int c = 0; c < TK / 32; ++c) tmem_st16(t_p + c * 16, &r[c * 16]);
                    }
                    // ---- the reference moved at this tile: rescale the running output (its last P V has been waited for above) ----
                    if (j > 0 && __any_sync(0xffffffffu, rescale)) {
                        if constexpr (!kOwnO && (!kSmemQ || kFirstRef)) {  // (returns at once; without it ptxas spills in the gathered kernels)
                            ok = mbar_wait_warp(smem_u32(&bars.pv_done[x ^ 1]), ((gs - 1) >> 1) & 1, abortp);
                            if (!ok) break;
                            tc_fence_after();
                        }
#pragma unroll 1  // rare path: kept small
                        for (int c = 0; c < D / 32; ++c) {
                            uint32_t o[32];
                            tmem_ld32(t_o + c * 32, o);
                            tc_wait_ld();
#pragma unroll
                            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                            tmem_st32(t_o + c * 32, o);
                        }
                    }
                    tc_wait_st();
                    tc_fence_before();
                    mbar_arrive(smem_u32(&bars.p_ready[x]));
                    BSA_PH(6);
                    if (lane == 0) BSA_STAMP(2 + warp, gs, 3);
#ifdef BSA_PHASES
                    ++ph_n;
#endif
                    if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 16);
                }
                if (!ok) break;
                // ---- hand this warpgroup's row sums, expressed in the item's final reference, to the epilogue warpgroup ----
                {
                    const uint32_t gl = g + n - 1;  // last tile of the item
                    const bool owner = (gl & 1) == (uint32_t)x;
                    float m_final = m_know;
                    if (!kOwnO && !owner) {  // the other warpgroup took the last tile: its publish holds the final reference
                        ok = __all_sync(0xffffffffu,
                                        take_reference(gl, *reinterpret_cast<volatile uint32_t*>(&mref[x ^ 1][tw]), m_final));
                        if (!ok) break;
                    }
                    if (m_final != m_know) l *= ex2_approx(m_know - m_final);  // l = 0 whenever m_know = -inf
                    // the previous item's sums must have been read
                    ok = mbar_wait_warp(smem_u32(&bars.e_taken), (itn & 1) ^ 1, abortp);
                    if (!ok) break;
                    lfin[x][tw] = l;
                    if (kOwnO) mref[x][tw] = __float_as_uint(m_know);
                    else if (owner) mfin[tw] = m_final;
                    mbar_arrive(smem_u32(&bars.e_ready));
                    ++itn;
                    if (lane == 0) BSA_TRACE_POINT(2 + warp, tn, 30);
                }
                g += n;
                BSA_PH(7);  // item boundary: sums handed over, next item's first tile not yet waited for
            }
        }
#ifdef BSA_PHASES
        if (blockIdx.x == 1 && lane == 0) {
            for (int k = 0; k < 8; ++k) g_trace[2 + warp][k] = ph_acc[k];
            g_trace[2 + warp][8] = ph_n;
        }
#endif
    }

    tc_fence_before();
    __syncthreads();
    if (tid == 0 && abort_flag) atomicExch(&p.counters->status, (int)BSA_ERR_DEVICE_TIMEOUT);
    if (warp == 9) tmem_dealloc(tmem, kTmemCols);
#ifdef BSA_TRACE
    if (tid == 0 && blockIdx.x < 4096) g_cta_times[1][blockIdx.x] = (long long)globaltimer_ns();
#endif
}

// ------------------------------------------------------------------------------------------
// Split-K reduction (Section 4.3): partial states were stored as (normalised O_p, LSE_p), so
// rescaling to the common maximum, merging and normalising is
//     LSE = log sum_p exp(LSE_p),  O = sum_p exp(LSE_p - LSE) O_p,
// taken in fixed partition order (bitwise reproducible).  One CTA per split Q tile row.
// ------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(256) bsa_merge_kernel(const SplitRow* __restrict__ split_rows,
                                                         const PlanCountersDev* __restrict__ counters,
                                                         const float* __restrict__ ws_O, const float* __restrict__ ws_LSE,
                                                         __nv_bfloat16* __restrict__ O, float* __restrict__ LSE, int N,
                                                         int f16, long long o_head, long long o_row) {
    constexpr int GROUPS = D / 8;                   // 8 output columns (16 bytes of bf16 or fp16) per thread
    constexpr int CHUNKS = kTQ * GROUPS / 256;      // CTAs' worth of work per merged 128-row tile
    const int n_units = counters->nsplit_rows * CHUNKS;
    for (int cu = blockIdx.x; cu < n_units; cu += gridDim.x) {
        const SplitRow s = split_rows[cu / CHUNKS];
        const int nparts = s.nparts & 0xffff, stride = s.nparts >> 16;
        const int u = (cu % CHUNKS) * 256 + threadIdx.x;
        const int r = u / GROUPS, gcol = (u % GROUPS) * 8;
        const int row = s.q_tile * kTQ + r;
        if (row >= N) continue;
        // all partial LSEs of the row first (independent loads), then the weights, then the weighted sum
        float lse_p[32];
        float m = -INFINITY;
#pragma unroll 4
        for (int q = 0; q < nparts; ++q) {
            lse_p[q & 31] = ws_LSE[(size_t)(s.ws_slot + q * stride) * kTQ + r];
            m = fmaxf(m, lse_p[q & 31]);
        }
        const float m_use = (m == -INFINITY) ? 0.f : m;
        float tot = 0.f;
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int q = 0; q < nparts; ++q) {
            const size_t slot = (size_t)(s.ws_slot + q * stride);
            const float w = __expf(lse_p[q & 31] - m_use);
            tot += w;
            const float4* src = reinterpret_cast<const float4*>(ws_O + (slot * kTQ + r) * D + gcol);
            const float4 a = src[0], b = src[1];
            acc[0] = fmaf(w, a.x, acc[0]); acc[1] = fmaf(w, a.y, acc[1]);
            acc[2] = fmaf(w, a.z, acc[2]); acc[3] = fmaf(w, a.w, acc[3]);
            acc[4] = fmaf(w, b.x, acc[4]); acc[5] = fmaf(w, b.y, acc[5]);
            acc[6] = fmaf(w, b.z, acc[6]); acc[7] = fmaf(w, b.w, acc[7]);
        }
        const float inv = (tot > 0.f) ? 1.f / tot : 0.f;
        uint4 v;
        if (f16) {
            v.x = pack_f16x2(acc[0] * inv, acc[1] * inv);
            v.y = pack_f16x2(acc[2] * inv, acc[3] * inv);
            v.z = pack_f16x2(acc[4] * inv, acc[5] * inv);
            v.w = pack_f16x2(acc[6] * inv, acc[7] * inv);
        } else {
            v.x = pack_bf16x2(acc[0] * inv, acc[1] * inv);
            v.y = pack_bf16x2(acc[2] * inv, acc[3] * inv);
            v.z = pack_bf16x2(acc[4] * inv, acc[5] * inv);
            v.w = pack_bf16x2(acc[6] * inv, acc[7] * inv);
        }
        *reinterpret_cast<uint4*>(O + ((size_t)s.head * o_head + (size_t)row * o_row) + gcol) = v;
        if (gcol == 0) LSE[(size_t)s.head * N + row] = (tot > 0.f) ? m_use + logf(tot) : -INFINITY;
    }
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// bf16 [heads][N][d] viewed as a 3-D tensor {d, N, heads}; box = {64, rows, 1}; rows beyond N read as zero.
// `nhd`: the tensor is stored [N][heads][d] instead (token-major); only the two byte strides change.
bool encode_map(CUtensorMap* m, const void* base, int64_t N, int heads, int d, int box_rows, bool f16, bool nhd) {
    EncodeTiledFn enc = get_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)N, (cuuint64_t)heads};
    cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)N * (cuuint64_t)d * 2};
    if (nhd) {
        strides[0] = (cuuint64_t)heads * (cuuint64_t)d * 2;
        strides[1] = (cuuint64_t)d * 2;
    }
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return enc(m, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims,
               strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same tensor as {64 columns, N rows, d/64 column groups, heads}; box = {64, rows, d/64, 1}: one copy lands all
// 64-column sub-tiles of a row block back to back (the [sub-tile][row][64] layout the MMA descriptors address).
// `col_groups` > 0: that many sub-tiles per copy instead of all d/64.
bool encode_map4(CUtensorMap* m, const void* base, int64_t N, int heads, int d, int box_rows, bool f16, bool nhd,
                 int col_groups = 0) {
    EncodeTiledFn enc = get_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[4] = {64, (cuuint64_t)N, (cuuint64_t)(d / 64), (cuuint64_t)heads};
    cuuint64_t strides[3] = {(cuuint64_t)d * 2, 128, (cuuint64_t)N * (cuuint64_t)d * 2};
    if (nhd) {
        strides[0] = (cuuint64_t)heads * (cuuint64_t)d * 2;
        strides[2] = (cuuint64_t)d * 2;
    }
    cuuint32_t box[4] = {64, (cuuint32_t)box_rows, (cuuint32_t)(col_groups > 0 ? col_groups : d / 64), 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    return enc(m, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims,
               strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D, int TK, int KERNEL, int G = 1>
cudaError_t launch_attn(const ForwardArgs& a, const AttnParams& p, cudaStream_t stream, const char** err) {
    CUtensorMap tq, tk, tv;
    const bool ok_maps = (KERNEL == 4)
                             ? (encode_map4(&tq, a.Q, a.g.N, a.g.H, D, kTQ, a.f16, a.nhd) &&
                                encode_map4(&tk, a.K, a.g.N_kv, a.g.H, D, TK / G, a.f16, a.nhd, G > 1 ? 1 : D / 64) &&
                                encode_map4(&tv, a.V, a.g.N_kv, a.g.H, D, TK / G, a.f16, a.nhd))
                             : (encode_map(&tq, a.Q, a.g.N, a.g.H, D, kTQ, a.f16, a.nhd) &&
                                encode_map(&tk, a.K, a.g.N_kv, a.g.H, D, TK, a.f16, a.nhd) &&
                                encode_map(&tv, a.V, a.g.N_kv, a.g.H, D, TK, a.f16, a.nhd));
    if (!ok_maps) {
        *err = "cuTensorMapEncodeTiled failed";
        return cudaErrorInvalidValue;
    }
    const int smem = attention_smem_bytes(D, TK, a.stages, KERNEL);
    if (a.f16 && (KERNEL == 1 || KERNEL == 2)) {  // not instantiated for half inputs (eligibility says so too)
        *err = "fp16 inputs need a single-tile, ping-pong or row-block plan";
        return cudaErrorInvalidValue;
    }
    // largest size already allowed, per instantiation and per device (the attribute belongs to the device's copy of
    // the kernel); concurrent first calls may both set it, which is harmless
    static std::atomic<int> attr_bytes_dev[kMaxDevices];
    const int dev = (a.device >= 0 && a.device < kMaxDevices) ? a.device : 0;
    if (smem > attr_bytes_dev[dev].load(std::memory_order_relaxed)) {
        cudaError_t e;
        if constexpr (KERNEL == 0 || KERNEL == 3) {
            e = cudaFuncSetAttribute(bsa_attention_kernel<D, TK, KERNEL == 3, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(bsa_attention_kernel<D, TK, KERNEL == 3, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        }
        else if constexpr (KERNEL == 1)
            e = cudaFuncSetAttribute(bsa_attention_pair_kernel<D, TK>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        else if constexpr (KERNEL == 2)
            e = cudaFuncSetAttribute(bsa_attention_cs_kernel<D, TK>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        else {
            const auto allow = [&](auto kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); };
            e = allow(bsa_attention_pp_kernel<D, false, G, true, false>);
            if (e == cudaSuccess) e = allow(bsa_attention_pp_kernel<D, true, G, true, false>);
            if constexpr (D != 64 || G != 2) {
                if (e == cudaSuccess) e = allow(bsa_attention_pp_kernel<D, false, G, false, true>);
            }
            if constexpr (D != 64) {
                if (e == cudaSuccess) e = allow(bsa_attention_pp_kernel<D, true, G, false, false>);
                if constexpr (G != 4)
                    if (e == cudaSuccess) e = allow(bsa_attention_pp_kernel<D, false, G, false, false>);
            }
        }
        if (e != cudaSuccess) {
            *err = "cudaFuncSetAttribute(max dynamic shared memory)";
            return e;
        }
        attr_bytes_dev[dev].store(smem, std::memory_order_relaxed);
    }
    int grid = a.num_sms < a.max_items ? a.num_sms : a.max_items;
    if (grid < 1) grid = 1;
    if constexpr (KERNEL == 0 || KERNEL == 3) {
        constexpr int threads = KERNEL == 3 ? kThreads + 32 : kThreads;
        if (a.f16)
            bsa_attention_kernel<D, TK, KERNEL == 3, true><<<grid, threads, smem, stream>>>(tq, tk, tv, p);
        else
            bsa_attention_kernel<D, TK, KERNEL == 3, false><<<grid, threads, smem, stream>>>(tq, tk, tv, p);
    }
    else if constexpr (KERNEL == 1)
        bsa_attention_pair_kernel<D, TK><<<grid, kPairThreads, smem, stream>>>(tq, tk, tv, p);
    else if constexpr (KERNEL == 2)
        bsa_attention_cs_kernel<D, TK><<<grid, kCsThreads, smem, stream>>>(tq, tk, tv, p);
    else {
        // The ping-pong kernel waits for its predecessor itself (grid_dependency_wait), so it may be scheduled while
        // the task-organisation kernel is still sorting: its launch latency and prologue overlap that kernel.
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3((unsigned)kPpThreads);
        cfg.dynamicSmemBytes = (size_t)smem;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const auto launch = [&](auto kernel) { return cudaLaunchKernelEx(&cfg, kernel, tq, tk, tv, p); };
        cudaError_t le = cudaErrorInvalidValue;
        // (at d = 128 the K producer of the short form relies on the two K tiles; tiles of two entries at d = 64 and of four at
        // d = 128 have one long form each, which serves them all: see choose_list_form)
        const bool short_form = D == 64 ? (G == 2 || !a.first_refs) : (a.short_lists && p.stages == 2 && p.stages_v > 2);
        const bool first_refs = !short_form && !a.f16 && (a.first_refs || G == 4);
        if (first_refs)  // whole waves of CTAs, of at most kRedoBits rounds each (max_items bounds the list's length)
            cfg.gridDim.x = (unsigned)(((int64_t)a.max_items + (int64_t)kRedoBits * grid - 1) / ((int64_t)kRedoBits * grid) * grid);
        if (short_form) {
            le = a.f16 ? launch(bsa_attention_pp_kernel<D, true, G, true, false>) : launch(bsa_attention_pp_kernel<D, false, G, true, false>);
        } else if (first_refs) {
            if constexpr (D != 64 || G != 2) le = launch(bsa_attention_pp_kernel<D, false, G, false, true>);
        } else if constexpr (D != 64) {
            if (a.f16) le = launch(bsa_attention_pp_kernel<D, true, G, false, false>);
            else if constexpr (G != 4) le = launch(bsa_attention_pp_kernel<D, false, G, false, false>);
        }
        count_launch();
        return le;
    }
    count_launch();
    return cudaGetLastError();
}

}  // namespace

bool encode_kv_map(CUtensorMap* m, const void* base, int64_t N, int heads, int d, int box_rows, bool f16, bool nhd) {
    return encode_map4(m, base, N, heads, d, box_rows, f16, nhd);
}

// Shared-memory budget: 227 KB per CTA minus each kernel's static shared memory (barriers, exchange
// buffer), which the compiler rounds up to the 1024-byte alignment of the dynamic part.
static int static_smem_bytes(int kernel) { return (kernel == 2 || kernel == 4) ? 3072 : 1024; }

static int kv_buffers_that_fit(int d, int T_KV, int kernel) {
    const int q = (kernel == 1 || (kernel == 4 && d == 64) ? 2 : 1) * kTQ * d * 2;  // two Q slots (kernel 1) or buffers
    const int kv = T_KV * d * 2;
    return (232448 - static_smem_bytes(kernel) - q) / kv;
}

static void split_stages(int total, int kernel, int* nk, int* nv) {
    if (kernel == 4) {
        // a K tile lives for one tile period (load -> its Q K^T), a V tile for about three (load -> its P V): two K
        // buffers measured as fast as three, so V gets three fifths
        *nk = total * 2 / 5;
        if (*nk < 2) *nk = 2;
    } else {
        *nk = total / 2;  // V is held one step longer than K, it gets the odd buffer
    }
    *nv = total - *nk;
    if (*nk > kMaxStages) *nk = kMaxStages;
    if (*nv > kMaxStages) *nv = kMaxStages;
}

int attention_max_stages(int d, int T_KV, int kernel) {
    if (kernel == 4) T_KV = kPpTK;
    if (kernel == kKernelRowBlock) return (d <= 128 && T_KV <= rb_max_chunk(d)) ? 2 : 0;  // rings of two slots and more per warp, see there
    if (d == 256 && !((kernel == 0 || kernel == 3) && T_KV == 64)) return 0;  // see launch_forward
    const int nb = kv_buffers_that_fit(d, T_KV, kernel);
    if (kernel == 1 || kernel == 4) return nb > 2 * kMaxStages ? 2 * kMaxStages : nb;  // total K + V buffers
    const int s = nb / 2;
    return s > kMaxStages ? kMaxStages : s;
}

int attention_smem_bytes(int d, int T_KV, int stages, int kernel) {
    if (kernel == 4) T_KV = kPpTK;
    const int q = (kernel == 1 || (kernel == 4 && d == 64) ? 2 : 1) * kTQ * d * 2;
    const int kv = T_KV * d * 2;
    int need = q + ((kernel == 1 || kernel == 4) ? stages : 2 * stages) * kv;
    // more than half of the SM's shared memory, so exactly one CTA (and one 512-column TMEM allocation) per SM
    if (need < 120 * 1024) need = 120 * 1024;
    return need;
}

#if defined(BSA_TRACE) || defined(BSA_PHASES)
extern "C" __attribute__((visibility("default"))) int bsa_debug_trace_copy(long long* host, int role) {
    if (role >= 100)  // 100 / 101: CTA entry / exit times
        return (int)cudaMemcpyFromSymbol(host, g_cta_times, sizeof(long long) * 4096, sizeof(long long) * 4096 * (role - 100));
    return (int)cudaMemcpyFromSymbol(host, g_trace, sizeof(long long) * 4096, sizeof(long long) * 4096 * role);
}
#endif

// Test hooks: the limit of the bounded device waits, and the withheld arrival described at g_withhold_arrival.
extern "C" __attribute__((visibility("default"))) bsa_status_t bsa_debug_set_wait_limit(long long cycles) {
    const long long v = cycles > 0 ? cycles : 2000000000ll;
    return cudaMemcpyToSymbol(ptx::g_wait_limit_cycles, &v, sizeof v) == cudaSuccess ? BSA_OK : BSA_ERR_CUDA;
}
extern "C" __attribute__((visibility("default"))) bsa_status_t bsa_debug_withhold_arrival(int on) {
    const int v = on ? 1 : 0;
    return cudaMemcpyToSymbol(g_withhold_arrival, &v, sizeof v) == cudaSuccess ? BSA_OK : BSA_ERR_CUDA;
}

cudaError_t launch_forward(const ForwardArgs& a, cudaStream_t stream, const char** err_detail) {
    AttnParams p;
    p.items = a.items;
    p.tile_col = a.tile_col;
    p.tile_member = a.tile_member;
    p.counters = a.counters;
    p.O = reinterpret_cast<__nv_bfloat16*>(a.O);
    p.LSE = a.LSE;
    p.ws_O = a.ws_O;
    p.ws_LSE = a.ws_LSE;
    const int bits = a.g.sQ128 * a.g.sK;
    p.full_member = (bits >= 64) ? ~0ull : ((1ull << bits) - 1ull);
    p.N = (int32_t)a.g.N;
    p.Nkv = (int32_t)a.g.N_kv;
    p.o_head = a.nhd ? (int64_t)a.d : (int64_t)a.g.N * a.d;
    p.o_wide = (reinterpret_cast<uintptr_t>(a.O) & 31) == 0;
    p.o_row = a.nhd ? (int64_t)a.g.H * a.d : (int64_t)a.d;
    p.lgBQ = (a.g.sQ128 > 1) ? a.g.lgBQ : 31;
    p.lgBKV = (a.g.sK > 1) ? a.g.lgBKV : 31;
    if (a.kernel == 4) {  // columns of a tile that share a membership bit
        p.lgBKV = -a.g.lgSK;
        while ((1 << (p.lgBKV + a.g.lgSK)) < a.g.T_KV) ++p.lgBKV;
    }
    p.sK = a.g.sK;
    p.lgSK = a.g.lgSK;
    p.stages = a.stages;
    p.stages_v = a.stages;
    if (a.kernel == 1 || a.kernel == 4) split_stages(a.stages, a.kernel, &p.stages, &p.stages_v);
    p.scale_log2 = (float)(1.4426950408889634 / sqrt((double)a.d));
    cudaError_t e;
    if (a.kernel == kKernelRowBlock) return launch_forward_rb(a, stream, err_detail);
    const int key = a.kernel * 1000 + a.d + a.g.T_KV / 64;  // kernel, d, T_KV
    if (key == 128 + 2) e = launch_attn<128, 128, 0>(a, p, stream, err_detail);
    else if (key == 128 + 1) e = launch_attn<128, 64, 0>(a, p, stream, err_detail);
    else if (key == 64 + 2) e = launch_attn<64, 128, 0>(a, p, stream, err_detail);
    else if (key == 64 + 1) e = launch_attn<64, 64, 0>(a, p, stream, err_detail);
    else if (key == 1000 + 128 + 2) e = launch_attn<128, 128, 1>(a, p, stream, err_detail);
    else if (key == 1000 + 128 + 1) e = launch_attn<128, 64, 1>(a, p, stream, err_detail);
    else if (key == 1000 + 64 + 2) e = launch_attn<64, 128, 1>(a, p, stream, err_detail);
    else if (key == 1000 + 64 + 1) e = launch_attn<64, 64, 1>(a, p, stream, err_detail);
    else if (key == 2000 + 128 + 2) e = launch_attn<128, 128, 2>(a, p, stream, err_detail);
    else if (key == 2000 + 128 + 1) e = launch_attn<128, 64, 2>(a, p, stream, err_detail);
    else if (key == 2000 + 64 + 2) e = launch_attn<64, 128, 2>(a, p, stream, err_detail);
    else if (key == 2000 + 64 + 1) e = launch_attn<64, 64, 2>(a, p, stream, err_detail);
    else if (key == 3000 + 128 + 2) e = launch_attn<128, 128, 3>(a, p, stream, err_detail);
    else if (key == 3000 + 128 + 1) e = launch_attn<128, 64, 3>(a, p, stream, err_detail);
    else if (key == 3000 + 64 + 2) e = launch_attn<64, 128, 3>(a, p, stream, err_detail);
    else if (key == 3000 + 64 + 1) e = launch_attn<64, 64, 3>(a, p, stream, err_detail);
    // d = 256: the output accumulator takes 256 of the 512 tensor-memory columns, which leaves room for the two score
    // buffers only where P is written in place over S (the single-tile kernels), with 64-key tiles
    else if (key == 256 + 1) e = launch_attn<256, 64, 0>(a, p, stream, err_detail);
    else if (key == 3000 + 256 + 1) e = launch_attn<256, 64, 3>(a, p, stream, err_detail);
    else if (key == 4000 + 128 + 2) e = launch_attn<128, kPpTK, 4>(a, p, stream, err_detail);
    else if (key == 4000 + 64 + 2) e = launch_attn<64, kPpTK, 4>(a, p, stream, err_detail);
    // narrower entries: two of 64 keys or four of 32 to a tile
    else if (key == 4000 + 128 + 1) e = launch_attn<128, kPpTK, 4, 2>(a, p, stream, err_detail);
    else if (key == 4000 + 128 && a.g.T_KV == 32) e = launch_attn<128, kPpTK, 4, 4>(a, p, stream, err_detail);
    else if (key == 4000 + 64 + 1) e = launch_attn<64, kPpTK, 4, 2>(a, p, stream, err_detail);
    else if (key == 4000 + 64 && a.g.T_KV == 32) e = launch_attn<64, kPpTK, 4, 4>(a, p, stream, err_detail);
    else {
        *err_detail = "no kernel for this (d, T_KV)";
        return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    if (a.has_split) e = launch_merge(a, stream);
    return e;
}

// Split-K reduction alone (also the merge-only test hook: the workspace then holds an earlier forward's partials).
cudaError_t launch_merge(const ForwardArgs& a, cudaStream_t stream) {
    const long long o_head = a.nhd ? (long long)a.d : (long long)a.g.N * a.d;
    const long long o_row = a.nhd ? (long long)a.g.H * a.d : (long long)a.d;
    // one CTA per 256 (row, 8-column) units of a merged tile, grid-strided beyond 8 waves
    const long long want = (long long)a.max_split_rows * (kTQ * (a.d / 8) / 256);
    int grid = want < 8ll * a.num_sms ? (int)want : 8 * a.num_sms;
    if (grid < 1) grid = 1;
    if (a.d == 256)
        bsa_merge_kernel<256><<<grid, 256, 0, stream>>>(a.split_rows, a.counters, a.ws_O, a.ws_LSE,
                                                        reinterpret_cast<__nv_bfloat16*>(a.O), a.LSE, (int)a.g.N, a.f16, o_head, o_row);
    else if (a.d == 128)
        bsa_merge_kernel<128><<<grid, 256, 0, stream>>>(a.split_rows, a.counters, a.ws_O, a.ws_LSE,
                                                        reinterpret_cast<__nv_bfloat16*>(a.O), a.LSE, (int)a.g.N, a.f16, o_head, o_row);
    else
        bsa_merge_kernel<64><<<grid, 256, 0, stream>>>(a.split_rows, a.counters, a.ws_O, a.ws_LSE,
                                                       reinterpret_cast<__nv_bfloat16*>(a.O), a.LSE, (int)a.g.N, a.f16, o_head, o_row);
    count_launch();
    return cudaGetLastError();
}

}  // namespace bsa
