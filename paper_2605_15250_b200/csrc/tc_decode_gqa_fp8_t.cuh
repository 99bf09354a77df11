// GQA-path split-KV flash decoding over an FP8 (E4M3) expanded cache with the TOKENS on the MMA's M axis (Eq. (mha)): the
// transposed products of tc_decode_gqa_t.cuh with the operand formats of tc_decode_gqa_fp8.cuh.
//
//   S^T = K Q^T     M = 128 tokens, N = R query rows, K = 192     (A = K tile, B = Q, both K-major; 6 MMAs of K = 32)
//   O^T = V^T P^T   M = 128 value columns, N = 32,    K = 128 tokens (A = V tile read MN-major, B = P^T rows; 4 MMAs)
//
// The tensor core does the method's FLOPs and not 128/R times as many: the row-replicating kernel is bound by the board's power
// (a fourfold product at 32 rows per group, a sixteenfold one at 8), this one by the cache stream.  Whole steps, us back to back,
// row-replicating -> this kernel, both in turn on one GPU: 64 x 4096 rows, 128 heads, s_q = 2 142.8 -> 116.0, s_q = 1 145.3 -> 103.9;
// 64 x 512-20000 rows, 32 heads 310.0 -> 221.5; four sequences of 3001 rows, 128 heads, s_q = 2 17.1 -> 16.2, s_q = 1 16.4 -> 14.6.
// Only where no CTA has more than one tile and 32 rows is the other one ahead (one sequence of 300 rows, s_q = 2: 11.1 and 11.8).
//
//   * A tile is 256 tokens, two halves of 128 that are loaded, multiplied and released by themselves (a ring of five halves,
//     40 KB each): what the softmax warps pay per tile -- barrier wake-ups, the vote, the hand-over of P^T -- is as long as the
//     work on 128 tokens of one byte.
//   * Sixteen softmax warps: two per half, TMEM lane quadrant and half of the query rows.  A thread owns one token and R/2 rows.
//   * References (m_ref) are those of the E4M3 kernels: one is put kF8Bias binades below the maximum that raised it and raised when
//     a score exceeds it by more than kF8Grow; whether any does is one barrier.red per tile behind a piece's first.  E4M3 reaches
//     2^-10, 16 binades below such a maximum, and what is smaller loses its bits, so ONE key that holds most of a row's weight costs
//     the tail of every token under its reference.  A row therefore has one reference, one row sum and one accumulator of O^T per
//     GROUP of tokens, as it has in the replicas of the row-replicating kernel, and the groups are weighed against each other in
//     fp32 at the end of a piece.  A group is the 32 tokens of a warp with 32 query rows (a k-step of P V is exactly one half's TMEM
//     quadrant: eight groups, four replicas there), its lower or upper 16 tokens with 16 (sixteen groups, eight or sixteen replicas
//     there).  With one reference per row, one key with 0.8 of the weight of 32768 rows gave errors of twice the tolerance.
//     A raise is passed on through shared memory, since a warp reads one lane quadrant of O^T only.
//   * P^T rows are 32 bytes per token (32-byte swizzle).  With 16 query rows the lower 16 tokens of a warp fill the lower half of
//     their rows and the upper 16 the upper half, the other half stays zero: a group each in the lower and upper 16 columns of O^T.
//   * Issuer and producer run converged (tc_common.cuh).
#pragma once
#include "common.cuh"
#include "sched.cuh"
#include "tc_common.cuh"
#include "tc_decode_absorb_fp8.cuh"  // kDescHiSw64
#include "tc_decode_gqa_fp8.cuh"     // GqaFp8Params, references, E4M3 helpers
#include "tc_decode_gqa_t.cuh"       // descriptor of MN-major rows, warp reductions

namespace gqla {
namespace tc {

template <int R>
struct GqaFp8TSmem {
    static constexpr int kQcBytes = R * 128;                 // R rows x 128 E4M3 (K_C part), 128-byte swizzle
    static constexpr int kQrBytes = R * 64;                  // R rows x 64 E4M3 (RoPE part), 64-byte swizzle
    static constexpr int kQBytes = kQcBytes + kQrBytes;
    static constexpr int kQRegion = (kQBytes + 1023) / 1024 * 1024;
    static constexpr int kKcBytes = 16384;                   // 128 tokens x 128
    static constexpr int kKrBytes = 8192;                    // 128 tokens x 64
    static constexpr int kVBytes = 16384;                    // 128 tokens x 128
    static constexpr int kStageBytes = kKcBytes + kKrBytes + kVBytes;
    static constexpr int kStages = 5;                        // halves of a tile
    static constexpr int kPRow = 32;                         // one token's probabilities
    static constexpr int kPBuf = 256 * kPRow;
    static constexpr int kOffStage = kQRegion;
    static constexpr int kOffP = kOffStage + kStages * kStageBytes;
    // Tables by column of the 8 x 32 columns of O^T (accumulator, column in it), i.e. by (group of tokens, query row):
    static constexpr int kCols = 8 * 32;
    static constexpr int kOffSum = kOffP + 2 * kPBuf;        // [kCols] row sums at a piece's end, maxima of a raise before; the plan scratch
    static constexpr int kOffRef = kOffSum + kCols * 4;      // [kCols] references
    static constexpr int kOffWeight = kOffRef + kCols * 4;   // [kCols] factors of a raise; the groups' weights in the output
    static constexpr int kOffScale = kOffWeight + kCols * 4; // [R] score scales of the piece's query rows
    static constexpr int kOffRow = kOffScale + R * 4;        // [R] row maxima of the piece's first tile
    static constexpr int kOffRaised = kOffRow + R * 4;       // [16] softmax warps that raised references
    static constexpr int kTileBytes = kOffRaised + 16 * 4;
    // q_full q_empty o_free kfull[5] vfull[5] kempty[5] vempty[5] s_full[2] p_ready[2] pv_done[2]
    static constexpr int kNumBars = 3 + 4 * kStages + 6;
    static constexpr int kSoftmaxWarps = 16;
    static constexpr int kThreads = 64 + 32 * kSoftmaxWarps;
    static constexpr int kTotal = kTileBytes + kNumBars * 8 + 16;
    static_assert(R == 16 || R == 32, "query rows are padded to 16 or 32");
    static_assert(kCols >= 3 * 32 + 4, "plan scratch must fit in the table of sums");
    static_assert(kTotal <= 232448, "shared memory budget of one CTA");
    static_assert(OneCtaPerSM<kTotal>::value, "");
};

// kind::f8f6f4 with descriptors as (low word, constant high word).
__device__ __forceinline__ void umma_f8_ss_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                              uint32_t idesc, uint32_t accumulate, uint32_t on) {
    asm volatile(
        "{\n\t.reg .b64 da, db;\n\t.reg .pred p, e;\n\t"
        "mov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\tsetp.ne.b32 p, %6, 0;\n\tsetp.ne.b32 e, %7, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], da, db, %5, p;\n\t}" ::"r"(d_tmem),
        "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate), "r"(on)
        : "memory");
}

// A group's first reference is that of the largest maximum among its row's groups on the piece's first tile, but at most this far
// above its own: the maximum of 16 or 32 tokens is soon outgrown by the 2.75 binades between kF8Bias and kF8Grow, and a raise costs
// 1.5 us (64 x 4096 rows, s_q = 2: raises on 63 % of the tiles and 180 us a step without this; 3 % with it, 116 us).  The group of
// the row's largest key keeps its full reach, one with a smaller maximum 14 of its 16 binades.
constexpr float kF8FirstUp = 2.0f;
// Floats as integers of the same order, and back.
__device__ __forceinline__ int float_order(float x) {
    const int i = __float_as_int(x);
    return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float float_unorder(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }
// A group that has no reference yet: finite, so that scores below every float still have the probability zero and not NaN.
constexpr float kF8NoRef = -FLT_MAX;

// N floats, N a multiple of 4, to and from 16-byte aligned shared memory.
template <int N>
__device__ __forceinline__ void store_row(float* dst, const float* v) {
#pragma unroll
    for (int c = 0; c < N; c += 4) *reinterpret_cast<float4*>(dst + c) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
}

template <int N>
__device__ __forceinline__ void load_row(float* v, const float* src) {
#pragma unroll
    for (int c = 0; c < N; c += 4) {
        const float4 a = *reinterpret_cast<const float4*>(src + c);
        v[c] = a.x; v[c + 1] = a.y; v[c + 2] = a.z; v[c + 3] = a.w;
    }
}

template <int R>
__global__ void __launch_bounds__(GqaFp8TSmem<R>::kThreads, 1)
decode_gqa_fp8_t_kernel(const GqaFp8Params p, const __grid_constant__ CUtensorMap tmQc, const __grid_constant__ CUtensorMap tmQr,
                        const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmR,
                        const __grid_constant__ CUtensorMap tmV) {
    using L = GqaFp8TSmem<R>;
    constexpr int NS = L::kStages;
    constexpr int RW = R / 2;   // query rows of a softmax thread
    constexpr int EW = RW / 2;  // rows that a warp stores
    constexpr int G = R;        // tokens (lanes of a warp) that share a reference
    constexpr int kGroups = L::kCols / R;
    constexpr int kSmT = 32 * L::kSoftmaxWarps;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* tiles = smem_raw;
    if ((smem_u32(tiles) & 1023u) != 0) {  // swizzled tiles need 1 KB alignment
        if (threadIdx.x == 0 && p.status != nullptr) atomicCAS(p.status, 0, kStatusTimeout | (15 << 8));
        return;
    }
    uint8_t* qc_smem = tiles;
    uint8_t* qr_smem = tiles + L::kQcBytes;
    uint8_t* stage0 = tiles + L::kOffStage;
    uint8_t* p_smem = tiles + L::kOffP;
    float* sm_sum = reinterpret_cast<float*>(tiles + L::kOffSum);
    float* sm_ref = reinterpret_cast<float*>(tiles + L::kOffRef);
    float* sm_w = reinterpret_cast<float*>(tiles + L::kOffWeight);
    float* sm_max = sm_sum;  // a tile's maxima
    float* sm_scale = reinterpret_cast<float*>(tiles + L::kOffScale);
    int* sm_row = reinterpret_cast<int*>(tiles + L::kOffRow);
    int* sm_raised = reinterpret_cast<int*>(tiles + L::kOffRaised);
    uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + L::kTileBytes);
    uint64_t* q_full = bars + 0;
    uint64_t* q_empty = bars + 1;
    uint64_t* o_free = bars + 2;
    uint64_t* kfull = bars + 3;
    uint64_t* vfull = kfull + NS;
    uint64_t* kempty = vfull + NS;
    uint64_t* vempty = kempty + NS;
    uint64_t* s_full = vempty + NS;   // [2]
    uint64_t* p_ready = s_full + 2;   // [2]
    uint64_t* pv_done = p_ready + 2;  // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + L::kNumBars);
    volatile int32_t* abort_flag = reinterpret_cast<volatile int32_t*>(tmem_slot + 1);

    // TMEM columns: two score buffers of 2 x R columns (a half each), then the eight 32-column output accumulators
    constexpr uint32_t kColS = 0, kColO = 4 * R;
    constexpr uint32_t kTmemCols = 512;
    static_assert(kColO + L::kCols <= kTmemCols, "");

    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const Abort ab{abort_flag, p.status};

    if (threadIdx.x == 0) {
        for (int i = 0; i < L::kNumBars; ++i) {
            const bool per_warp = &bars[i] == o_free || &bars[i] == &p_ready[0] || &bars[i] == &p_ready[1];
            mbar_init(&bars[i], per_warp ? L::kSoftmaxWarps : 1);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, kTmemCols);
        tmem_relinquish();
    }

    pdl_launch_dependents();
    if (warp == 0 && elect_one()) {
        tma_prefetch_desc(&tmQc);
        tma_prefetch_desc(&tmQr);
        tma_prefetch_desc(&tmK);
        tma_prefetch_desc(&tmR);
        tma_prefetch_desc(&tmV);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = warp_uniform(*tmem_slot);
    pdl_wait();  // set-up is done (behind the preceding kernel's tail); everything below reads the caller's tensors
    const int j = blockIdx.x % p.g;
    const int unit = blockIdx.x / p.g;
    Walker walk;
    if (p.balanced) {
        const BalancedStart st = balanced_prepass(p.seqlens, p.B, p.S, unit, p.W, reinterpret_cast<int32_t*>(sm_sum), L::kThreads);
        walk.init_balanced(p.seqlens, p.B, p.S, unit, p.W, st);
    } else {
        walk.init_fixed(p.seqlens, p.B, p.S, unit / p.S, unit % p.S);
    }
    Piece pc;    // its n_tiles counts halves
    int gt = 0;  // tiles walked so far: S / P buffer = gt & 1, phase = (gt >> 1) & 1
    int pi = 0;  // non-empty pieces walked so far

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        const uint32_t e = elect_one();
        int s = 0;
        uint32_t ph = 1;  // parity that means "slot is free"
        bool ok = true;
        auto load_q = [&](uint8_t* dst, const CUtensorMap* m, int32_t x, int32_t b) {
            asm volatile(
                "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %7, 0;\n\t@e cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], "
                "[%1, {%3, %4, %5, %6}], [%2];\n\t}" ::"r"(smem_u32(dst)),
                "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(q_full)), "r"(x), "r"(0), "r"(j), "r"(b * p.s_q), "r"(e)
                : "memory");
        };
        while (ok && warp_all(walk.next(pc))) {
            const int n_halves = warp_uniform(pc.n_tiles);
            if (n_halves == 0) continue;
            int64_t half_row = p.rows.row(pc.b, pc.tok_begin);
            for (int t = 0; t < n_halves; ++t) {
                uint8_t* st = stage0 + s * L::kStageBytes;
                const int32_t row = warp_uniform((int32_t)half_row);
                if (t + 1 < n_halves)
                    half_row = p.rows.paged() ? p.rows.row(pc.b, pc.tok_begin + (t + 1) * 128) : half_row + 128;
                if (!(ok = warp_all(mbar_wait(&kempty[s], ph, ab, 1)))) break;
                mbar_expect_tx(&kfull[s], L::kKcBytes + L::kKrBytes, e);
                tma_load_3d(st, &tmK, 0, j, row, &kfull[s], e);
                tma_load_2d(st + L::kKcBytes, &tmR, 0, row, &kfull[s], e);
                // Q of the piece goes out behind its first K: that one only needs a free slot, Q needs every Q K^T of the
                // previous piece to have completed
                if (t == 0) {
                    if (pi > 0 && !(ok = warp_all(mbar_wait(q_empty, (pi - 1) & 1, ab, 13)))) break;
                    mbar_expect_tx(q_full, L::kQBytes, e);
                    const int32_t b = warp_uniform(pc.b);
                    load_q(qc_smem, &tmQc, 0, b);
                    load_q(qr_smem, &tmQr, 128, b);
                }
                if (!(ok = warp_all(mbar_wait(&vempty[s], ph, ab, 2)))) break;
                mbar_expect_tx(&vfull[s], L::kVBytes, e);
                tma_load_3d(st + L::kKcBytes + L::kKrBytes, &tmV, 0, j, row, &vfull[s], e);
                if (++s == NS) { s = 0; ph ^= 1; }
            }
            ++pi;
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t e = elect_one();
        constexpr uint32_t idesc_qk = idesc_e4m3(128, R, 0, 0);   // S^T: A = K tile (K-major), B = Q (K-major)
        constexpr uint32_t idesc_pv = idesc_e4m3(128, 32, 1, 1);  // O^T: A = V tile read MN-major, B = P^T rows (MN-major)
        const uint32_t qc_lo = desc_lo(desc_kmajor_sw128(smem_u32(qc_smem))), qr_lo = desc_lo(desc_kmajor_sw64(smem_u32(qr_smem)));
        const uint64_t pd0 = desc_mnmajor_rows(smem_u32(p_smem), L::kPRow);
        int ks = 0, vs = 0;
        uint32_t kph = 0, vph = 0;
        auto issue_qk = [&](int n, int halves) -> bool {
#pragma unroll 1
            for (int h = 0; h < halves; ++h) {
                if (!warp_all(mbar_wait_fast(&kfull[ks], kph, ab, 3))) return false;
                tc_fence_after();
                const uint32_t st = smem_u32(stage0 + ks * L::kStageBytes);
                const uint32_t d = tmem_base + kColS + (uint32_t)((n & 1) * 2 + h) * R;
                const uint32_t k_lo = desc_lo(desc_kmajor_sw128(st)), r_lo = desc_lo(desc_kmajor_sw64(st + L::kKcBytes));
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)  // K_C part: 128 elements = 4 x 32
                    umma_f8_ss_lo(d, k_lo + ((kk * 32) >> 4), kDescHiSw128, qc_lo + ((kk * 32) >> 4), kDescHiSw128, idesc_qk, kk != 0, e);
#pragma unroll
                for (int kk = 0; kk < 2; ++kk)  // k_R part: 64 elements = 2 x 32
                    umma_f8_ss_lo(d, r_lo + ((kk * 32) >> 4), kDescHiSw64, qr_lo + ((kk * 32) >> 4), kDescHiSw64, idesc_qk, 1, e);
                umma_commit(&kempty[ks], e);
                if (++ks == NS) { ks = 0; kph ^= 1; }
            }
            umma_commit(&s_full[n & 1], e);
            return true;
        };
        bool ok = true;
        while (ok && warp_all(walk.next(pc))) {
            const int n_halves = warp_uniform(pc.n_tiles);
            if (n_halves == 0) continue;
            const int nt = (n_halves + 1) >> 1;
            if (!(ok = warp_all(mbar_wait(q_full, pi & 1, ab, 4)))) break;
            tc_fence_after();
            if (!(ok = issue_qk(gt, n_halves > 1 ? 2 : 1))) break;
            for (int t = 0; t < nt && ok; ++t) {
                const int n = gt + t;
                if (t + 1 < nt) {
                    if (!(ok = issue_qk(n + 1, n_halves - 2 * (t + 1) > 1 ? 2 : 1))) break;
                } else {
                    umma_commit(q_empty, e);
                }
                if (!(ok = warp_all(mbar_wait_fast(&p_ready[n & 1], (n >> 1) & 1, ab, 5)))) break;
                if (t == 0 && pi > 0 && !(ok = warp_all(mbar_wait(o_free, (pi - 1) & 1, ab, 14)))) break;
                const int halves = n_halves - 2 * t > 1 ? 2 : 1;
#pragma unroll 1
                for (int h = 0; h < halves; ++h) {
                    if (!(ok = warp_all(mbar_wait_fast(&vfull[vs], vph, ab, 6)))) break;
                    tc_fence_after();
                    const uint64_t vd =
                        desc_mnmajor_sw128(smem_u32(stage0 + vs * L::kStageBytes + L::kKcBytes + L::kKrBytes), 16384);
                    const uint32_t p_lo = (uint32_t)pd0 + (((n & 1) * L::kPBuf + h * 128 * L::kPRow) >> 4);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)  // 32 tokens per step, an accumulator each: rows [32 kk, +32) of V and of P^T
                        umma_f8_ss_lo(tmem_base + kColO + (uint32_t)(h * 4 + kk) * 32, (uint32_t)vd + ((kk * 4096) >> 4),
                                      (uint32_t)(vd >> 32), p_lo + ((kk * 32 * L::kPRow) >> 4), (uint32_t)(pd0 >> 32), idesc_pv,
                                      t != 0, e);
                    umma_commit(&vempty[vs], e);
                    if (++vs == NS) { vs = 0; vph ^= 1; }
                }
                if (ok) umma_commit(&pv_done[n & 1], e);
            }
            gt += nt;
            ++pi;
        }
    } else {
        // ------------------------------------------------------------------ softmax: one TMEM lane = one token per thread
        const int q = warp & 3;
        const int sub = (warp - 2) >> 3;         // which half of the tile
        const int half = ((warp - 2) >> 2) & 1;  // which half of the query rows: [r0, +RW)
        const int r0 = half * RW;
        const int e0 = r0 + sub * EW;            // rows this warp stores: [e0, +EW)
        const int tl = sub * 128 + q * 32 + lane;  // token within the tile
        const int si = threadIdx.x - 64;           // index among the softmax threads
        // this thread's rows in the tables: accumulator (half of the tile, quadrant), with 16 rows its lower or upper columns
        static_assert(G / RW == 2 && kGroups * EW == 64, "");
        const int col0 = (sub * 4 + q) * 32 + (R == 32 ? 0 : lane & 16) + r0;
        const uint32_t lane_base = tmem_base + ((uint32_t)(q * 32) << 16);
        const int hshift = __ffs(p.hpg_box) - 1;  // hpg_box is a power of two: query position of row r = r >> hshift
        const int r_hi = p.s_q << hshift;
        const uint32_t pswz = ((uint32_t)(tl * L::kPRow) >> 7) & 1u;  // XOR of the row's 16-byte chunks
        const uint32_t pchunk = R == 32 ? (uint32_t)half : (uint32_t)lane >> 4;  // 16-byte chunk that holds this thread's rows
        uint8_t* prow = p_smem + tl * L::kPRow + ((pchunk ^ pswz) << 4) + (R == 32 ? 0 : half * 8);
        float m_ref[RW], l[RW];  // of rows r0 .. r0 + RW - 1 and this thread's group, in log2 units

        if (R == 16 && half == 0) {  // the other 16 bytes of every P^T row stay zero
#pragma unroll
            for (int s = 0; s < 2; ++s)
                *reinterpret_cast<uint4*>(p_smem + s * L::kPBuf + tl * L::kPRow + ((pchunk ^ 1u ^ pswz) << 4)) = make_uint4(0, 0, 0, 0);
        }

        while (walk.next(pc)) {
            const int32_t T = p.seqlens[pc.b];
            const int64_t slot0 = (int64_t)pc.b * p.S;
            GQLA_DEBUG_CHECK(pc.b >= 0 && pc.b < p.B, p.status, 32);
            GQLA_DEBUG_CHECK(pc.n_tiles == 0 || (pc.k >= 0 && pc.k < p.S), p.status, 33);
            GQLA_DEBUG_CHECK(pc.tok_begin >= 0 && pc.tok_begin <= pc.tok_end && pc.tok_end <= (T > 0 ? T : 0), p.status, 34);
            const int64_t out_row0 = ((slot0 + pc.k) * p.s_q) * p.h_q + (int64_t)j * p.hpg;
            if (si < R) {  // thread r of the first R: row r's empty slots and its score scale
                const int r = si, pq = r >> hshift, il = r & (p.hpg_box - 1);
                const bool row_valid = il < p.hpg && pq < p.s_q;
                if (row_valid)
                    for (int kk = pc.fill_begin; kk < pc.fill_end; ++kk)
                        p.lse_part[((slot0 + kk) * p.s_q + pq) * p.h_q + (int64_t)j * p.hpg + il] = -INFINITY;
                sm_row[r] = float_order(-INFINITY);
                // softmax scale x log2(e) x the query row's quantisation scale
                sm_scale[r] = p.scale_log2 *
                              (row_valid ? p.q_scale[((int64_t)pc.b * p.s_q + pq) * p.h_q + (int64_t)j * p.hpg + il] : 1.f);
            }
            if (pc.n_tiles == 0 && p.balanced) continue;
            named_bar_sync(1, kSmT);  // the scales are there
#pragma unroll
            for (int r = 0; r < RW; ++r) { m_ref[r] = kF8NoRef; l[r] = 0.f; }
            const int nt = (pc.n_tiles + 1) >> 1;
            bool ok = true;

            for (int t = 0; t < nt && ok; ++t) {
                const int n = gt + t;
                const int s = n & 1;
                // A wait that fails raises the CTA's abort flag; the warps agree on leaving at the next barrier below
                // (a warp that left the loop on its own would strand the others in that barrier).
                bool okl = __all_sync(0xffffffffu, mbar_wait_fast(&s_full[s], (n >> 1) & 1, ab, 7));
                // P^T buffer s was last read by P.V(n-2)
                if (okl && t > 1) okl = __all_sync(0xffffffffu, mbar_wait_fast(&pv_done[s], ((n - 2) >> 1) & 1, ab, 8));
                tc_fence_after();
                // rows this thread's token is visible to: the token at absolute position ta is seen by query positions
                // pq >= s_q - (T - ta); padding positions see nothing
                const int ta = pc.tok_begin + t * 256 + tl;
                const int pq_min = p.s_q - (T - ta) > 0 ? p.s_q - (T - ta) : 0;
                const int r_lo = ta < pc.tok_end ? (pq_min << hshift) : R;
                const bool full = __all_sync(0xffffffffu, r_lo == 0 && r_hi == R && okl);  // every row sees every token
                uint32_t x[RW];
                if (okl) {
                    tmem_ld<RW>(lane_base + kColS + (uint32_t)(2 * s + sub) * R + r0, x);
                    tmem_wait_ld();
                }
                float d[RW];
                auto against = [&](const float* ref) {  // scores against references (log2 units), -inf where the token is not visible
                    load_row<RW>(d, sm_scale + r0);
#pragma unroll
                    for (int c = 0; c < RW; ++c) d[c] = fmaf(__uint_as_float(x[c]), d[c], ref != nullptr ? -ref[c] : 0.f);
                    if (!full) {
#pragma unroll
                        for (int c = 0; c < RW; ++c)
                            if (!(okl && r0 + c >= r_lo && r0 + c < r_hi)) d[c] = -INFINITY;
                    }
                };
                auto group_maxima = [&]() {  // of d, into the table
                    warp_reduce_scatter<RW, G>(d, lane, [](float a, float b) { return fmaxf(a, b); });
                    if (lane % 2 == 0) sm_max[col0 + lane % G / 2] = d[0];
                };
                if (t == 0) {
                    // a piece's first tile gives the references: the maxima meet in shared memory
                    against(nullptr);
                    group_maxima();
                    if (lane % 2 == 0) atomicMax(sm_row + r0 + lane % G / 2, float_order(d[0]));
                    if (bar_or(!okl, kSmT)) { ok = false; break; }
                    load_row<RW>(d, sm_max + col0);
#pragma unroll
                    for (int c = 0; c < RW; c += 4) {
                        const int4 top4 = *reinterpret_cast<const int4*>(sm_row + r0 + c);
                        const int top[4] = {top4.x, top4.y, top4.z, top4.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            m_ref[c + i] = d[c + i] > kF8NoRef ? fminf(float_unorder(top[i]), d[c + i] + kF8FirstUp) - kF8Bias : kF8NoRef;
                    }
                    against(m_ref);
                } else {
                    against(m_ref);
                    float top = -INFINITY;
#pragma unroll
                    for (int c = 0; c < RW; ++c) top = fmaxf(top, d[c]);
                    if (bar_or(top > kF8Grow || !okl, kSmT)) {
                        const bool raise = __any_sync(0xffffffffu, top > kF8Grow);
                        if (raise) {
                            against(nullptr);
                            group_maxima();
                            __syncwarp();
                            load_row<RW>(d, sm_max + col0);  // (of this warp's own groups)
#pragma unroll
                            for (int c = 0; c < RW; ++c) {
                                const bool need = d[c] > m_ref[c] + kF8Grow;
                                const float mn = need ? d[c] - kF8Bias : m_ref[c];
                                d[c] = need ? ex2(m_ref[c] - mn) : 1.f;  // ex2(-FLT_MAX - ..) = 0 on first use
                                l[c] *= d[c];
                                m_ref[c] = mn;
                            }
                            if (lane % G == 0) store_row<RW>(sm_w + col0, d);
                        }
                        if (lane == 0) sm_raised[(sub * 2 + half) * 4 + q] = raise;
                        if (bar_or(!okl, kSmT)) { ok = false; break; }  // the factors are there; leaving is agreed on (tc_common.cuh)
                        // O^T may be rescaled only between P.V(n-1) completing and P.V(n) being issued
                        if (!__all_sync(0xffffffffu, mbar_wait(&pv_done[(n - 1) & 1], ((n - 1) >> 1) & 1, ab, 8))) {
                            okl = false;  // noticed by everybody at the next barrier
                        } else {
                            tc_fence_after();
                            // the four warps of a lane quadrant take two of the eight accumulators each, of these the
                            // columns of the warps that raised
#pragma unroll 1
                            for (int i = 0; i < 8; ++i) {
                                const int a = (sub * 2 + half) * 2 + (i >> 2), h = (i >> 1) & 1;
                                if (!sm_raised[((a >> 2) * 2 + h) * 4 + (a & 3)]) continue;
                                const int c = a * 32 + (R == 32 ? h * 16 + (i & 1) * 8 : h * 8 + (i & 1) * 16);
                                uint32_t o[8];
                                tmem_ld<8>(lane_base + kColO + c, o);
                                tmem_wait_ld();
#pragma unroll
                                for (int k = 0; k < 8; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) * sm_w[c + k]);
                                tmem_st<8>(lane_base + kColO + c, o);
                            }
                            tmem_wait_st();
                        }
                        against(m_ref);
                    }
                }
                // probabilities of this token -> its row of P^T (a group that has no reference yet sees nothing: d = -inf there)
                uint32_t pk[RW / 4];
#pragma unroll
                for (int c = 0; c < RW; c += 4) {
                    float ex[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        ex[i] = ex2(d[c + i]);
                        l[c + i] += ex[i];
                    }
                    pk[c / 4] = pack_e4m3x4(ex[0], ex[1], ex[2], ex[3]);
                }
                if constexpr (R == 32)
                    *reinterpret_cast<uint4*>(prow + s * L::kPBuf) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                else
                    *reinterpret_cast<uint2*>(prow + s * L::kPBuf) = make_uint2(pk[0], pk[1]);
                fence_proxy_async_smem();  // generic-proxy writes of P^T -> visible to the tensor core
                tc_fence_before();
                __syncwarp();
                if (lane == 0 && okl) mbar_arrive(&p_ready[s]);
            }

            // -------------------------------------------------------------- row sums over the tokens, then the output
            // (neither the sums nor the weights need the last P.V: they are made while it runs)
            warp_reduce_scatter<RW, G>(l, lane, [](float a, float b) { return a + b; });
            if (lane % 2 == 0) sm_sum[col0 + lane % G / 2] = l[0];
            if (lane % G == 0) store_row<RW>(sm_ref + col0, m_ref);
            named_bar_sync(1, kSmT);
            // the weights of this warp's EW rows in their kGroups groups, two a lane (the warps of the other quadrants write the
            // same values to the same places)
            constexpr int KB = 32 / EW;
            const int wi = lane / EW * R + e0 + lane % EW;
            const float m0 = sm_ref[wi], m1 = sm_ref[wi + KB * R];
            float M = fmaxf(m0, m1);
#pragma unroll
            for (int o = EW; o < 32; o *= 2) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
            const float w0 = m0 > kF8NoRef ? ex2(m0 - M) : 0.f, w1 = m1 > kF8NoRef ? ex2(m1 - M) : 0.f;
            float Lt = (m0 > kF8NoRef ? sm_sum[wi] * w0 : 0.f) + (m1 > kF8NoRef ? sm_sum[wi + KB * R] * w1 : 0.f);
#pragma unroll
            for (int o = EW; o < 32; o *= 2) Lt += __shfl_xor_sync(0xffffffffu, Lt, o);
            const bool seen = Lt > 0.f;
            const float inv = seen ? p.v_scale / Lt : 0.f;
            sm_w[wi] = seen ? w0 * inv : 0.f;
            sm_w[wi + KB * R] = seen ? w1 * inv : 0.f;
            __syncwarp();
            const int n_last = gt + nt - 1;
            if (nt > 0 && ok) ok = __all_sync(0xffffffffu, mbar_wait_fast(&pv_done[n_last & 1], (n_last >> 1) & 1, ab, 9));
            tc_fence_after();
            if (q == 0 && lane < EW) {
                const int r = e0 + lane, pq = r >> hshift, il = r & (p.hpg_box - 1);
                if (il < p.hpg && pq < p.s_q)
                    p.lse_part[out_row0 + (int64_t)pq * p.h_q + il] = ok && seen ? (M + log2f(Lt)) * 0.6931471805599453f : -INFINITY;
            }
            float acc[EW];
#pragma unroll
            for (int c = 0; c < EW; ++c) acc[c] = 0.f;
            if (nt > 0 && ok) {  // warp-uniform
#pragma unroll 1
                for (int k0 = 0; k0 < (pc.n_tiles > 1 ? kGroups : KB); k0 += KB) {  // (a single half: the other's accumulators hold anything)
                    uint32_t o[KB * EW];
#pragma unroll
                    for (int k = 0; k < KB; ++k) tmem_ld<EW>(lane_base + kColO + (k0 + k) * R + e0, o + k * EW);
                    tmem_wait_ld();
#pragma unroll
                    for (int k = 0; k < KB; ++k)
#pragma unroll
                        for (int c = 0; c < EW; c += 4) {
                            const float4 w = *reinterpret_cast<const float4*>(sm_w + (k0 + k) * R + e0 + c);
                            acc[c] = fmaf(__uint_as_float(o[k * EW + c]), w.x, acc[c]);
                            acc[c + 1] = fmaf(__uint_as_float(o[k * EW + c + 1]), w.y, acc[c + 1]);
                            acc[c + 2] = fmaf(__uint_as_float(o[k * EW + c + 2]), w.z, acc[c + 2]);
                            acc[c + 3] = fmaf(__uint_as_float(o[k * EW + c + 3]), w.w, acc[c + 3]);
                        }
                }
            }
#pragma unroll
            for (int c = 0; c < EW; ++c) {
                const int r = e0 + c, pq = r >> hshift, il = r & (p.hpg_box - 1);
                const bool some = __shfl_sync(0xffffffffu, inv, c) != 0.f;
                // a lane holds one value column of every row: 128 consecutive floats per row over the quadrants
                if (il < p.hpg && pq < p.s_q)  // padding rows are computed and dropped
                    p.o_part[(out_row0 + (int64_t)pq * p.h_q + il) * 128 + q * 32 + lane] = some ? acc[c] : 0.f;
            }
            named_bar_sync(1, kSmT);  // the tables may be rewritten by the next piece
            // O^T has been read: the next piece's first P.V may overwrite it
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(o_free);
            gt += nt;
            if (pc.n_tiles > 0) ++pi;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
}

}  // namespace tc
}  // namespace gqla
