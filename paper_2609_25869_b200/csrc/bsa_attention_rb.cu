// Row-block attention kernel: physical Q tiles of 16 rows (paper Section 4.2: the physical tile need not be the
// logical block; Section 4.4: a catalog holds several tile shapes per architecture).
//
// The tensor-memory kernels of bsa_attention.cu compute 128 query rows per MMA, so logical blocks of 16 to 64 rows
// are Coarsened onto them and every physical tile also computes the pairs of its inactive sub-blocks (4-5 times the
// active pairs on masks whose neighbouring row blocks select different columns).  This kernel keeps such masks at
// their own granularity instead: one WARP owns a 16-row fragment of a logical row block (a 16-row physical tile,
// Refined along Q for B_Q > 16) and walks that block's own KV tile list with the register-level tensor instruction
// mma.sync.m16n8k16 (bf16 or fp16 in, fp32 accumulate), FlashAttention-2 style:
//   * K and V are copied in steps of at most 32 keys into two 8 KB rings private to the warp, by TMA tiles (128-byte
//     swizzle) that one lane issues: K read back with ldmatrix, V with ldmatrix.trans; a ring slot is refilled as soon
//     as the warp has read it, so the next steps' copies are in flight during the arithmetic of the current one;
//   * S = Q K^T, online softmax with the running row maximum in the exp2 domain, P rounded to bf16 in registers
//     (the accumulator layout of two 8-key tiles is the A-operand layout of one 16-key step), O += P V;
//   * no block-level synchronisation: twelve independent warps per SM, each takes the next of the CTA's items when it is free.
// A block of 16 rows and 64 keys (d = 64) is 262 kflop on 16 KB of K and V, each byte used once: 133 clk of MMA per SM, and
// shared memory sees the bytes twice (copy in, ldmatrix).  The kernel takes 242 clk a block: tensor pipe 53 % busy, issue 44 %,
// its three warps per sub-partition mostly wait for the latency of their own instructions.  With per-thread cp.async copies
// of whole entries the load path stopped at about 41 B/clk per SM (bulk copies reach 80); now, on one GPU, 32768 tokens, 16
// heads, d = 64, (16,64) blocks, 15 % active in runs: 3.58 -> 2.77 ms; the same with 32-key entries 4.01 -> 2.94 ms, (32,32)
// blocks at d = 128 52 -> 40 ms; maxima agreed on only where one has moved, and items taken by free warps instead of a fixed
// share each: 2.82 -> 2.50, independent blocks at 15 % 2.48 -> 2.28, (16,16) blocks at 10 %, 16384 tokens, 4 heads
// 214 -> 170 us.  (Fragments loaded straight from global memory, no shared memory at all: 5.4 ms, the L1 miss path moves
// about 32 B/clk.  Fourteen warps: spills, 3.95.)
// The register-level instruction peaks at about a third of the tcgen05 rate on this GPU, so the kernel pays off only
// where Coarsening wastes more than that; the plan table decides per regime.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

#include <atomic>

#include "bsa_common.h"
#include "sm100_ptx.cuh"

namespace bsa {

using namespace ptx;

namespace {

constexpr int kRbWarps = 12;        // warps per CTA (one CTA per SM)
constexpr int kRbStageBytes = 8192; // one warp's K or V ring
constexpr unsigned kFullMask = 0xffffffffu;

struct RbParams {
    const __nv_bfloat16* Q;
    __nv_bfloat16* O;
    float* LSE;
    const WorkItem* items;
    const int32_t* tile_col;
    PlanCountersDev* counters;
    long long q_head, q_row;    // element strides of Q and O between heads / token rows
    int32_t N, Nkv;
    float scale_log2;           // log2(e) / sqrt(d)
};

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
// D (16x8, fp32) += A (16x16, row-major) * B (16x8, column-major); A and B bf16, or IEEE half with F16
template <bool F16>
__device__ __forceinline__ void mma_16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    if (F16)
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
    else
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
template <bool F16>
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {  // two fp32 -> the kernel's 16-bit element type
    uint32_t r;
    if (F16)
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    else
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Byte offset of 16-byte chunk `chunk` of row `row` in a ring slot of ROWS rows as the copy lays it out: 64-column
// halves one after the other, 128-byte rows, the chunk index XORed with the row's low three bits, so that the eight row
// addresses of an ldmatrix fall into eight different bank groups.
template <int ROWS>
__device__ __forceinline__ uint32_t swz(int row, int chunk) {
    return (uint32_t)((chunk >> 3) * (ROWS * 128) + row * 128 + (((chunk & 7) ^ (row & 7)) << 4));
}

// Keys per step: small enough that a ring holds two of them.
template <int D, int CK>
constexpr int kRbStep = (CK * D * 4 <= kRbStageBytes) ? CK : kRbStageBytes / (D * 4);

template <int D, int CK, bool F16>
__global__ void __launch_bounds__(kRbWarps * 32, 1)
bsa_attention_rb_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const RbParams p) {
    constexpr int KS = kRbStep<D, CK>;      // keys per step
    constexpr int SPE = CK / KS;            // steps per entry of the tile list
    constexpr int SLOT = KS * D * 2;        // bytes of a ring slot
    constexpr int NST = kRbStageBytes / SLOT;
    static_assert(KS % 16 == 0 && CK % KS == 0 && D % 64 == 0 && NST >= 2, "whole MMA steps");
    constexpr int NT_S = KS / 8;   // 8-key accumulator tiles of S
    constexpr int KS_QK = D / 16;  // 16-wide steps over the head dimension
    constexpr int KS_PV = KS / 16; // 16-key steps of P V
    constexpr int NT_O = D / 8;    // 8-column accumulator tiles of O
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t bars[kRbWarps][2 * NST];  // K slots, then V slots: the copy has landed
    __shared__ uint32_t abort_flag;
    __shared__ int next_round;  // of the CTA's items: the next one no warp has taken
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const uint32_t sK = smem_u32(smem + warp * 2 * kRbStageBytes), sV = sK + kRbStageBytes;
    const uint32_t bK = smem_u32(&bars[warp][0]), bV = bK + NST * 8;
    if (smem_u32(smem) & 1023u) {  // never expected; fail with a status instead of corrupting tiles
        if (threadIdx.x == 0) atomicExch(&p.counters->status, (int)BSA_ERR_CUDA);
        return;
    }
    if (threadIdx.x == 0) abort_flag = next_round = 0;
    if (lane == 0) {
        for (int i = 0; i < 2 * NST; ++i) mbar_init(bK + i * 8, 1);
        fence_mbar_init();
    }
    __syncthreads();
    volatile uint32_t* abortp = &abort_flag;

    const int n_items = p.counters->nitems;
    // The CTA's items (dealt in alternating directions per round of the list, longest first) go to whichever warp is free.
    // A fixed share per warp left the SM to its last busy warps: with row lists of 14 to 431 entries (32768 tokens, 16
    // heads, runs) the SMs' sums of fixed shares differ by 19 %, a warp's from the mean by 24 %.
    auto take_item = [&]() -> int {
        int k = 0;
        if (lane == 0) k = atomicAdd(&next_round, 1);
        k = __shfl_sync(kFullMask, k, 0);
        return k * (int)gridDim.x + ((k & 1) ? ((int)gridDim.x - 1 - (int)blockIdx.x) : (int)blockIdx.x);
    };
    auto load_record = [&](int idx) { return __ldg(reinterpret_cast<const int4*>(p.items + (idx < n_items ? idx : 0))); };
    const float c2 = p.scale_log2;
    int slot = 0;          // ring slot of the current step (the same for K and V)
    uint32_t phase = 0;    // its barriers' phase
    bool ok = true;

    int idx = take_item();
    int4 record = load_record(idx);
    while (idx < n_items) {
        const int head = record.x, q_tile = record.y, tile_begin = record.z, tile_end = record.w;
        const int row0 = q_tile * 16;
        const int r_lo = row0 + g, r_hi = row0 + g + 8;
        __nv_bfloat16* o_lo = p.O + (long long)head * p.q_head + (long long)r_lo * p.q_row;
        __nv_bfloat16* o_hi = p.O + (long long)head * p.q_head + (long long)r_hi * p.q_row;
        if (tile_end <= tile_begin) {  // no active column: zero output, LSE = -inf
#pragma unroll
            for (int n = 0; n < NT_O; ++n) {
                if (r_lo < p.N) *reinterpret_cast<uint32_t*>(o_lo + n * 8 + 2 * t) = 0u;
                if (r_hi < p.N) *reinterpret_cast<uint32_t*>(o_hi + n * 8 + 2 * t) = 0u;
            }
            if (t == 0) {
                if (r_lo < p.N) p.LSE[(long long)head * p.N + r_lo] = -INFINITY;
                if (r_hi < p.N) p.LSE[(long long)head * p.N + r_hi] = -INFINITY;
            }
            idx = take_item();
            record = load_record(idx);
            continue;
        }
        const int n_steps = (tile_end - tile_begin) * SPE;
        auto first_key = [&](int st) { return __ldg(p.tile_col + tile_begin + st / SPE) * CK + (st % SPE) * KS; };
        auto copy_in = [&](uint32_t dst, const CUtensorMap* map, uint32_t bar, int key0) {
            mbar_arrive_expect_tx(bar, SLOT);
            tma_load_4d(dst, map, bar, 0, key0, 0, head);
        };
        // the first steps' copies are on their way while the Q fragment is loaded
        if (lane == 0) {
            int sl = slot;
            for (int st = 0; st < NST && st < n_steps; ++st) {
                const int key0 = first_key(st);
                copy_in(sK + sl * SLOT, &tmK, bK + sl * 8, key0);
                copy_in(sV + sl * SLOT, &tmV, bV + sl * 8, key0);
                if (++sl == NST) sl = 0;
            }
        }
        const int last_key = __ldg(p.tile_col + tile_end - 1) * CK;  // columns ascend: only the last entry can be ragged
        int key_next = (NST < n_steps) ? first_key(NST) : 0;         // of the step to copy next
        // Q fragment (A operand, row-major 16 x 16 per step): rows g and g+8, columns 2t, 2t+1 and 8 further
        uint32_t qa[KS_QK][4];
        {
            const __nv_bfloat16* q_lo = p.Q + (long long)head * p.q_head + (long long)r_lo * p.q_row;
            const __nv_bfloat16* q_hi = p.Q + (long long)head * p.q_head + (long long)r_hi * p.q_row;
#pragma unroll
            for (int ks = 0; ks < KS_QK; ++ks) {
                const int c = ks * 16 + 2 * t;
                qa[ks][0] = (r_lo < p.N) ? __ldg(reinterpret_cast<const uint32_t*>(q_lo + c)) : 0u;
                qa[ks][1] = (r_hi < p.N) ? __ldg(reinterpret_cast<const uint32_t*>(q_hi + c)) : 0u;
                qa[ks][2] = (r_lo < p.N) ? __ldg(reinterpret_cast<const uint32_t*>(q_lo + c + 8)) : 0u;
                qa[ks][3] = (r_hi < p.N) ? __ldg(reinterpret_cast<const uint32_t*>(q_hi + c + 8)) : 0u;
            }
        }
        float o[NT_O][4];
#pragma unroll
        for (int n = 0; n < NT_O; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
        float m_lo = -INFINITY, m_hi = -INFINITY;  // running row maxima, exp2 domain (score * c2)
        float l_lo = 0.f, l_hi = 0.f;              // this thread's share of the row sums

        for (int st = 0; st < n_steps; ++st) {
            const bool more = st + NST < n_steps;
            if (st == n_steps - NST || (st == 0 && n_steps < NST)) {  // nothing left to copy: the next item's record instead
                idx = take_item();
                record = load_record(idx);
            }
            const int key_in = key_next;
            if (st + NST + 1 < n_steps) key_next = first_key(st + NST + 1);
            const uint32_t cK = sK + slot * SLOT, cV = sV + slot * SLOT;
            // ---- S = Q K^T ----
            ok = mbar_wait_warp(bK + slot * 8, phase, abortp);
            if (!ok) break;
            float s[NT_S][4];
#pragma unroll
            for (int n = 0; n < NT_S; ++n) s[n][0] = s[n][1] = s[n][2] = s[n][3] = 0.f;
#pragma unroll
            for (int np = 0; np < NT_S / 2; ++np) {
#pragma unroll
                for (int ks = 0; ks < KS_QK; ++ks) {
                    // four 8x8 matrices: keys np*16 + {0..7, 8..15} x head-dim columns ks*16 + {0..7, 8..15}
                    const int key = np * 16 + ((lane >> 4) << 3) + (lane & 7);
                    const int chunk = ks * 2 + ((lane >> 3) & 1);
                    uint32_t b0, b1, b2, b3;
                    ldmatrix_x4(cK + swz<KS>(key, chunk), b0, b1, b2, b3);
                    mma_16816<F16>(s[2 * np], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], b0, b1);
                    mma_16816<F16>(s[2 * np + 1], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], b2, b3);
                }
            }
            __syncwarp();  // every lane has read the K slot
            if (more && lane == 0) copy_in(cK, &tmK, bK + slot * 8, key_in);
            // ---- online softmax ----
            if (st >= n_steps - SPE && last_key + CK > p.Nkv) {  // ragged last entry: keys at or beyond N_kv do not exist
#pragma unroll
                for (int n = 0; n < NT_S; ++n) {
                    const int kc = last_key + (st % SPE) * KS + n * 8 + 2 * t;
                    if (kc >= p.Nkv) s[n][0] = s[n][2] = -INFINITY;
                    if (kc + 1 >= p.Nkv) s[n][1] = s[n][3] = -INFINITY;
                }
            }
            float mx_lo = max3(s[0][0], s[0][1], s[1][0]), mx_hi = max3(s[0][2], s[0][3], s[1][2]);
            mx_lo = fmaxf(mx_lo, s[1][1]);
            mx_hi = fmaxf(mx_hi, s[1][3]);
#pragma unroll
            for (int n = 2; n < NT_S; ++n) {
                mx_lo = max3(mx_lo, s[n][0], s[n][1]);
                mx_hi = max3(mx_hi, s[n][2], s[n][3]);
            }
            mx_lo *= c2;
            mx_hi *= c2;
            // The running maxima have moved for some row of the fragment in about a third of the steps of a long list: only
            // then do the four lanes of a row have to agree, and the sums and the output to be rescaled.
            if (__any_sync(kFullMask, mx_lo > m_lo || mx_hi > m_hi)) {
                mx_lo = fmaxf(mx_lo, __shfl_xor_sync(kFullMask, mx_lo, 1));
                mx_hi = fmaxf(mx_hi, __shfl_xor_sync(kFullMask, mx_hi, 1));
                mx_lo = fmaxf(mx_lo, __shfl_xor_sync(kFullMask, mx_lo, 2));
                mx_hi = fmaxf(mx_hi, __shfl_xor_sync(kFullMask, mx_hi, 2));
                const float mn_lo = fmaxf(m_lo, mx_lo), mn_hi = fmaxf(m_hi, mx_hi);
                const float a_lo = (m_lo == -INFINITY) ? 0.f : ex2(m_lo - mn_lo);
                const float a_hi = (m_hi == -INFINITY) ? 0.f : ex2(m_hi - mn_hi);
                m_lo = mn_lo;
                m_hi = mn_hi;
                l_lo *= a_lo;
                l_hi *= a_hi;
#pragma unroll
                for (int n = 0; n < NT_O; ++n) {
                    o[n][0] *= a_lo;
                    o[n][1] *= a_lo;
                    o[n][2] *= a_hi;
                    o[n][3] *= a_hi;
                }
            }
            const float nm_lo = (m_lo == -INFINITY) ? 0.f : -m_lo, nm_hi = (m_hi == -INFINITY) ? 0.f : -m_hi;
            const uint64_t c22 = pack_f32x2(c2, c2), nm_lo2 = pack_f32x2(nm_lo, nm_lo), nm_hi2 = pack_f32x2(nm_hi, nm_hi);
            uint64_t sum_lo2 = pack_f32x2(0.f, 0.f), sum_hi2 = sum_lo2;
            uint32_t pa[KS_PV][4];  // P as the A operand of P V
#pragma unroll
            for (int n = 0; n < NT_S; ++n) {
                float x0, x1, x2, x3;
                unpack_f32x2(fma_f32x2(pack_f32x2(s[n][0], s[n][1]), c22, nm_lo2), x0, x1);
                unpack_f32x2(fma_f32x2(pack_f32x2(s[n][2], s[n][3]), c22, nm_hi2), x2, x3);
                const float p0 = ex2(x0), p1 = ex2(x1), p2 = ex2(x2), p3 = ex2(x3);
                sum_lo2 = add_f32x2(sum_lo2, pack_f32x2(p0, p1));
                sum_hi2 = add_f32x2(sum_hi2, pack_f32x2(p2, p3));
                pa[n >> 1][(n & 1) * 2 + 0] = pack_bf16<F16>(p0, p1);
                pa[n >> 1][(n & 1) * 2 + 1] = pack_bf16<F16>(p2, p3);
            }
            {
                float a0, a1, b0, b1;
                unpack_f32x2(sum_lo2, a0, a1);
                unpack_f32x2(sum_hi2, b0, b1);
                l_lo += a0 + a1;
                l_hi += b0 + b1;
            }
            // ---- O += P V ----
            ok = mbar_wait_warp(bV + slot * 8, phase, abortp);
            if (!ok) break;
#pragma unroll
            for (int ks = 0; ks < KS_PV; ++ks) {
#pragma unroll
                for (int nd = 0; nd < NT_O / 2; ++nd) {
                    // four 8x8 matrices, transposed on the way: keys ks*16 + {0..7, 8..15} x columns nd*16 + {0..7, 8..15}
                    const int key = ks * 16 + (((lane >> 3) & 1) << 3) + (lane & 7);
                    const int chunk = nd * 2 + (lane >> 4);
                    uint32_t b0, b1, b2, b3;
                    ldmatrix_x4_trans(cV + swz<KS>(key, chunk), b0, b1, b2, b3);
                    mma_16816<F16>(o[2 * nd], pa[ks][0], pa[ks][1], pa[ks][2], pa[ks][3], b0, b1);
                    mma_16816<F16>(o[2 * nd + 1], pa[ks][0], pa[ks][1], pa[ks][2], pa[ks][3], b2, b3);
                }
            }
            __syncwarp();  // every lane has read the V slot
            if (more && lane == 0) copy_in(cV, &tmV, bV + slot * 8, key_in);
            if (++slot == NST) {
                slot = 0;
                phase ^= 1u;
            }
        }
        if (!ok) break;
        // ---- epilogue: row sums over the four lanes of a row, normalise, store ----
        l_lo += __shfl_xor_sync(kFullMask, l_lo, 1);
        l_hi += __shfl_xor_sync(kFullMask, l_hi, 1);
        l_lo += __shfl_xor_sync(kFullMask, l_lo, 2);
        l_hi += __shfl_xor_sync(kFullMask, l_hi, 2);
        const float inv_lo = (l_lo > 0.f) ? 1.f / l_lo : 0.f, inv_hi = (l_hi > 0.f) ? 1.f / l_hi : 0.f;
#pragma unroll
        for (int n = 0; n < NT_O; ++n) {
            if (r_lo < p.N) *reinterpret_cast<uint32_t*>(o_lo + n * 8 + 2 * t) = pack_bf16<F16>(o[n][0] * inv_lo, o[n][1] * inv_lo);
            if (r_hi < p.N) *reinterpret_cast<uint32_t*>(o_hi + n * 8 + 2 * t) = pack_bf16<F16>(o[n][2] * inv_hi, o[n][3] * inv_hi);
        }
        if (t == 0) {
            if (r_lo < p.N)
                p.LSE[(long long)head * p.N + r_lo] = (l_lo > 0.f) ? fmaf(m_lo, 0.6931471805599453f, logf(l_lo)) : -INFINITY;
            if (r_hi < p.N)
                p.LSE[(long long)head * p.N + r_hi] = (l_hi > 0.f) ? fmaf(m_hi, 0.6931471805599453f, logf(l_hi)) : -INFINITY;
        }
    }
    if (!ok) {  // a wait ran out: copies in flight land before the CTA's shared memory goes away
        if (lane == 0) atomicExch(&p.counters->status, (int)BSA_ERR_DEVICE_TIMEOUT);
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
}

template <int D, int CK, bool F16>
cudaError_t launch_rb_t(const ForwardArgs& a, const RbParams& p, cudaStream_t stream, const char** err) {
    constexpr int smem = kRbWarps * 2 * kRbStageBytes;
    static std::atomic<int> attr_set_dev[kMaxDevices];
    const int dev = (a.device >= 0 && a.device < kMaxDevices) ? a.device : 0;
    if (!attr_set_dev[dev].load(std::memory_order_relaxed)) {
        cudaError_t e = cudaFuncSetAttribute(bsa_attention_rb_kernel<D, CK, F16>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) {
            *err = "cudaFuncSetAttribute(max dynamic shared memory)";
            return e;
        }
        attr_set_dev[dev].store(1, std::memory_order_relaxed);
    }
    int grid = a.max_items < a.num_sms ? a.max_items : a.num_sms;  // (few items: one warp each on as many SMs as there are)
    if (grid < 1) grid = 1;
    CUtensorMap tk, tv;
    if (!encode_kv_map(&tk, a.K, a.g.N_kv, a.g.H, D, kRbStep<D, CK>, F16, a.nhd) ||
        !encode_kv_map(&tv, a.V, a.g.N_kv, a.g.H, D, kRbStep<D, CK>, F16, a.nhd)) {
        *err = "cuTensorMapEncodeTiled failed";
        return cudaErrorInvalidValue;
    }
    bsa_attention_rb_kernel<D, CK, F16><<<grid, kRbWarps * 32, smem, stream>>>(tk, tv, p);
    count_launch();
    return cudaGetLastError();
}
template <int D, int CK>
cudaError_t launch_rb(const ForwardArgs& a, const RbParams& p, cudaStream_t stream, const char** err) {
    return a.f16 ? launch_rb_t<D, CK, true>(a, p, stream, err) : launch_rb_t<D, CK, false>(a, p, stream, err);
}

}  // namespace

// Largest KV entry (keys) the row-block kernel takes for head dimension d.
int rb_max_chunk(int d) { return kRbStageBytes / (d * 2); }

cudaError_t launch_forward_rb(const ForwardArgs& a, cudaStream_t stream, const char** err_detail) {
    RbParams p;
    p.Q = reinterpret_cast<const __nv_bfloat16*>(a.Q);
    p.O = reinterpret_cast<__nv_bfloat16*>(a.O);
    p.LSE = a.LSE;
    p.items = a.items;
    p.tile_col = a.tile_col;
    p.counters = a.counters;
    p.q_head = a.nhd ? (long long)a.d : (long long)a.g.N * a.d;
    p.q_row = a.nhd ? (long long)a.g.H * a.d : (long long)a.d;
    p.N = (int32_t)a.g.N;
    p.Nkv = (int32_t)a.g.N_kv;
    p.scale_log2 = (float)(1.4426950408889634 / sqrt((double)a.d));
    const int key = a.d * 1000 + a.g.T_KV;
    if (key == 64 * 1000 + 64) return launch_rb<64, 64>(a, p, stream, err_detail);
    if (key == 64 * 1000 + 32) return launch_rb<64, 32>(a, p, stream, err_detail);
    if (key == 64 * 1000 + 16) return launch_rb<64, 16>(a, p, stream, err_detail);
    if (key == 128 * 1000 + 32) return launch_rb<128, 32>(a, p, stream, err_detail);
    if (key == 128 * 1000 + 16) return launch_rb<128, 16>(a, p, stream, err_detail);
    *err_detail = "no row-block kernel for this (d, T_KV)";
    return cudaErrorInvalidValue;
}

}  // namespace bsa
