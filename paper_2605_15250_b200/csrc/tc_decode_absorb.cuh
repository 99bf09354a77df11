// Absorb-path split-KV flash decoding on tcgen05 (Eq. (mqa), lines 3-5): a PAIR of CTAs (one
// 2-CTA cluster, cta_group::2 MMAs) works for one block of 128 query rows and walks the
// (sequence, split) pieces its plan gives it (sched.cuh): exactly one piece under the fixed plan,
// an equal share of the batch's 128-row tiles under the balanced plan (persistent pair).
//
//   S = Qh Kh^T    Qh: 128 rows (head, query) x 576,  Kh = [c ; k_R] rows of the latent cache
//   O = P  V       V = the first 512 columns of the same cache rows
//
// Why a pair: O for 128 rows x 512 fp32 columns is all 256 KB of one SM's tensor memory, leaving no
// room for S.  With a 2-CTA MMA of M = 128 each CTA holds 64 rows; its accumulators use all 128 TMEM
// lanes for half as many columns (lanes 0-63: columns [0, N/2), lanes 64-127: columns [N/2, N) of
// the same 64 rows), so O takes 256 columns and S (128 tokens) 64.  Each CTA also supplies half of
// every B operand from its own shared memory: 64 of the tile's 128 cache rows for S = Qh Kh^T, and
// 128 of every 256 latent columns for O = P V.  The cache is fetched from HBM once; the second
// operand shape comes out of L2 ([64 rows x 64 columns] 8 KB boxes, 128-byte swizzle).
//
// Staging: two rings per CTA, one of K groups (three 8 KB boxes = 192 columns of 64 rows) and one of
// V groups (two box pairs = one token half of a tile), each one tile deep (the V ring of column halves
// two), each filled by a producer warp of its own;
// the loads of tile t+1 are in flight while the MMAs of tile t run, and the K loads of the next piece
// while this piece is stored.
// The issuer and the producers run converged (tc_common.cuh): 64 x 4096 rows 85.2 -> 82.8 us at the power cap, 48 x 1000-9001
// rows at s_q = 2 153 -> 147, one of 777 rows 10.3 -> 9.8, small pages (32 x 300-8000 rows, pages of 64) 88.0 -> 83.3.
// Barriers are per group, not per box: every barrier operation of the issuing threads costs on the
// order of 100 cycles next to tensor-core operand traffic, and one MMA of this shape is only 32-64
// cycles of tensor work.
//
// Warp roles per CTA: warp 0 TMA producer of Q and K, warp 1 TMEM owner (+ MMA issuer in the leader CTA),
// warps 2-9 softmax, warp 10 TMA producer of V.  A softmax thread owns one TMEM lane = (row, token half)
// and one half of that lane's 64 score columns, so a row's 128 scores of a tile sit in four threads of
// four different warps; they share the tile maximum through shared memory and keep separate partial sums.
//
// Small pages (template parameter PG = rows of a box: 32 or 16; 0 = the form above).  A paged cache whose pages are
// no multiple of the 128-row tile is fetched in boxes of PG rows that no page boundary cuts (PG divides the page size
// and the tile's halves): the boxes of a group go out together, one lane of the producer warp each, after every lane has
// looked its page up; boxes behind the sequence's end start behind the cache's last row and are filled with zeros, and of the
// box that the end cuts V gets zeros behind it (load_cut_run): rows outside a sequence may hold anything.  Such
// calls keep 32-bit probabilities: P is split into three bf16 terms, which hold all of its 24 bits, and P V is issued for each of
// them.  The two further P buffers are paid for by a K ring of seven single column blocks in place of three groups of three and a
// V ring of three groups of 32 tokens in place of two of 64: P V takes three quarters of a tile's MMA time, so V streams through
// less, and all but two of the next tile's K blocks wait for their turn in shared memory (five K blocks and one tile of V: 99.4 us
// a step on the batch below instead of 96.3; nine blocks and two V groups 96.5).  The products of the second and third term go to
// accumulators of their own where tensor memory has room for them (half of O here, all of it in the tokens-on-M kernels): the
// tensor core truncates its running sums, so every further addition into one of them costs bits (relative to O about 1.7e-8 per
// 16 rows and term).  What bounds it: what the MMAs read through shared memory (with the loads 616 KB a tile and CTA; 504 with two
// terms, 392 in the form above); 96 us a step on 32 sequences of 300-8000 rows in pages of 64 rows, 128 heads.  Neither an issuer
// that polls for K groups and P alike nor P written by token halves while P V of the other half runs made it faster.
// Errors of the merged partials there, against 64 bits: 3.6e-6 of the 2-norm (two terms 3.8e-6, SIMT kernel 3.4e-7); of the step:
// 2.79e-3 with each of the three, from the roundings to bf16.  These calls ran one warp per query row on the SIMT kernel before,
// which read every cache row h_q times from L2: 13.7 ms for 32 sequences of 300-8000 rows in pages of 64 rows.
#pragma once
#include "common.cuh"
#include "sched.cuh"
#include "tc_common.cuh"

namespace gqla {
namespace tc {

struct AbsorbParams {
    int32_t B, S, s_q, h_q, rows_total /* s_q*h_q */, row_blocks /* ceil(rows_total/128) */;
    int32_t balanced, W;  // balanced plan: W pairs per row block, grid = 2 * W * row_blocks
    float scale_log2;
    RowMap rows;      // packed or paged (PG = 0: pages a multiple of 128 rows, pieces starting on tile boundaries)
    const int32_t* seqlens;
    float* o_part;    // [B, S, s_q*h_q, 512]
    float* lse_part;  // [B, S, s_q*h_q]
    __nv_bfloat16* o_final;  // not null: S = 1, fixed plan; the normalised output goes here as bf16 [B, s_q*h_q, 512]
                             // (o_part unused, lse_part may be null)
    int32_t* status;
    int32_t n_rows;   // rows of the cache (small pages: where the zero-filled boxes start)
    int32_t workers;  // column halves, balanced plan: worker ids launched per row block, the last of them stands for W - 1
};

template <int PG, bool HALF = false>
struct AbsorbSmemT {
    static constexpr int kBox = 8192;              // 64 rows x 64 bf16, 128-byte swizzle
    static constexpr int kQBytes = 9 * kBox;       // 64 query rows x 576
    static constexpr int kPTerms = PG != 0 ? 3 : 1;  // bf16 terms of a probability
    static constexpr int kPTerm = 2 * kBox;        // 64 rows x 128 tokens (two 64-token k-blocks)
    static constexpr int kPBytes = kPTerms * kPTerm;
    static constexpr int kKBlocks = PG != 0 ? 1 : 3;  // column blocks of a K group
    static constexpr int kKGroup = kKBlocks * kBox;   // of this CTA's 64 rows of a tile
    static constexpr int kVRows = PG != 0 ? 32 : 64;  // tokens of a V group
    static constexpr int kVBox = kVRows * 128;        // kVRows tokens x 64 latent columns
    static constexpr int kBlocks = HALF ? 1 : 2;      // blocks of 256 latent columns that a pair gives
    static constexpr int kVGroup = 2 * kBlocks * kVBox;  // kVRows tokens x this CTA's 128 columns of each block
    static constexpr int kNK = PG != 0 ? 7 : 3;    // ring of K groups (Qh Kh^T operand)
    static constexpr int kNV = PG != 0 ? 3 : (HALF ? 4 : 2);    // ring of V groups (P V operand)
    static constexpr int kOffK = kQBytes;
    static constexpr int kOffP = kOffK + kNK * kKGroup;
    static constexpr int kOffV = kOffP + kPBytes;
    static constexpr int kTileBytes = kOffV + kNV * kVGroup;
    // kfull[kNK] kempty[kNK] vfull[kNV] vempty[kNV] q_full q_empty o_free epi_done s_full[2] p_ready[2]
    // pv_done[2] xch[2] fin epi
    static constexpr int kNumBars = 2 * kNK + 2 * kNV + 14;
    static constexpr int kSoftmaxWarps = 8;
    static constexpr int kVProducerWarp = 2 + kSoftmaxWarps;  // behind the softmax warps
    static constexpr int kThreads = 96 + 32 * kSoftmaxWarps;
    // output staging for the epilogue (P and the V ring, idle once the last P.V of a piece has completed), padded pitches:
    // the final bf16 rows (64 x 1 KB) at once
    static constexpr int kOutPitch = 256 * 4 + 16;
    static_assert(64 * kOutPitch <= kPBytes + kNV * kVGroup, "output staging must fit in P + V ring");
    static constexpr int kWarpPitch = 64 * 4 + 16;  // fp32 partials: a softmax warp's 32 rows x 64 columns
    static_assert(8 * 32 * kWarpPitch <= kPBytes + kNV * kVGroup, "output staging must fit in P + V ring");
    // behind the barriers: tmem slot + abort flag (16 B), sm_max [2][4][64] (sm_l [4][64] and the plan
    // scratch reuse it).  No slack for re-aligning the base: the kernel checks the 1 KB alignment.
    static constexpr int kTotal = kTileBytes + kNumBars * 8 + 16 + 2 * 4 * 64 * 4;
    static_assert(2 * 4 * 64 >= kThreads + 4, "plan scratch must fit in sm_max");
    static_assert(kTotal <= 232448, "shared memory budget of one CTA");
    static_assert(OneCtaPerSM<kTotal>::value, "");
    static_assert(PG == 0 || PG == 32 || PG == 16, "");
    static_assert(!HALF || PG == 0, "small pages: both blocks");
};
using AbsorbSmem = AbsorbSmemT<0>;

constexpr uint32_t kAColO = 0;    // O: MMA m (latent columns [256m, 256m+256)) at TMEM columns [128m, 128m+128)
constexpr uint32_t kAColS = 256;  // two 64-column score buffers
constexpr uint32_t kAColRest = 384;  // small pages: the part of O's MMA 0 that the second and third terms of P give

// FINAL: the whole-sequence call (o_final set); a form of its own, so that neither output's registers weigh on the softmax
// loop of the other.
// HALF: a pair gives one block of 256 latent columns of O; two pairs (blockIdx / 2 even and odd) share a piece and both compute
// its scores.  For calls that leave at least half of the device idle (the rule stands in tc_dispatch.cuh): half of a pair's P V, V
// loads and output (an SM writes about 30 B a clock, 128 KB of partials are 2.3 us).  Whole steps, us: one sequence of 777 rows
// 22.5 -> 20.7, of 100 rows 20.9 -> 18.7, of 1500 rows at s_q = 2 25.3 -> 23.2; two of 300-900 rows 23.3 -> 21.0, four of 200-500
// rows 24.6 -> 22.5.
template <int PG, bool FINAL = false, bool HALF = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(AbsorbSmemT<PG, HALF>::kThreads, 1)
decode_absorb_tc_kernel(const AbsorbParams p, const __grid_constant__ CUtensorMap tmQ,
                        const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CutMaps<PG> cut_maps) {
    using L = AbsorbSmemT<PG, HALF>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* tiles = smem_raw;
    if ((smem_u32(tiles) & 1023u) != 0) {  // swizzled tiles need 1 KB alignment; same answer in both CTAs
        if (threadIdx.x == 0 && p.status != nullptr) atomicCAS(p.status, 0, kStatusTimeout | (15 << 8));
        return;
    }
    uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + L::kTileBytes);
    uint64_t* kfull = bars;
    uint64_t* kempty = kfull + L::kNK;
    uint64_t* vfull = kempty + L::kNK;
    uint64_t* vempty = vfull + L::kNV;
    uint64_t* q_full = vempty + L::kNV;
    uint64_t* q_empty = q_full + 1;    // every Qh Kh^T of a piece has completed: Q may be overwritten
    uint64_t* o_free = q_empty + 1;    // leader only: both CTAs' softmax warps have read O of a piece
    uint64_t* epi_done = o_free + 1;   // this CTA's output staging (P + V ring) is free again
    uint64_t* s_full = epi_done + 1;   // [2]
    uint64_t* p_ready = s_full + 2;    // [2] leader only: one arrival per softmax warp of the pair
    uint64_t* pv_done = p_ready + 2;   // [2]
    uint64_t* xch = pv_done + 2;       // [2] softmax warps of this CTA: per-tile max exchange
    uint64_t* fin = xch + 2;           //     the final partial-sum exchange of a piece
    uint64_t* epi = fin + 1;           //     and the step of the output staging (whole-sequence form)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + L::kNumBars);
    volatile int32_t* abort_flag = reinterpret_cast<volatile int32_t*>(tmem_slot + 1);
    float* sm_max = reinterpret_cast<float*>(tmem_slot + 4);  // [2][4][64] per-tile partial maxima
    // [4][64] final partial sums; written only after the last P.V of a piece, i.e. after every warp has
    // arrived on p_ready of its last tile and hence finished reading sm_max
    float* sm_l = sm_max;

    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t cta = cluster_ctarank();  // 0 = leader
    const Abort ab{abort_flag, p.status};

    if (threadIdx.x == 0) {
        for (int i = 0; i < L::kNumBars; ++i) {
            uint64_t* bar = &bars[i];
            const bool pair_wide = bar == &p_ready[0] || bar == &p_ready[1] || bar == o_free;
            const bool cta_wide = bar == &xch[0] || bar == &xch[1] || bar == fin || bar == epi || bar == epi_done;
            mbar_init(bar, pair_wide ? 2 * L::kSoftmaxWarps : (cta_wide ? L::kSoftmaxWarps : 1));
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc2(tmem_slot, 512);
        tmem_relinquish2();
    }

    pdl_launch_dependents();
    if (warp == 0 && elect_one()) {
        tma_prefetch_desc(&tmQ);
        tma_prefetch_desc(&tmC);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // both CTAs' barriers exist before any remote arrival
    tc_fence_after();
    const uint32_t tmem_base = warp_uniform(*tmem_slot);
    pdl_wait();  // set-up is done (behind the preceding kernel's tail); everything below reads the caller's tensors
    // the plan of this pair: row block rb, and either one (sequence, split) piece or worker w's share
    const int pair = HALF ? blockIdx.x >> 2 : blockIdx.x >> 1;
    const int blk0 = HALF ? (blockIdx.x >> 1) & 1 : 0;  // first block of 256 columns of this pair
    const int rb = pair % p.row_blocks;
    Walker walk;
    if (p.balanced) {
        int w = pair / p.row_blocks;
        if (HALF && w == p.workers - 1) w = p.W - 1;  // the workers in between have no tiles
        const BalancedStart st = balanced_prepass(p.seqlens, p.B, p.S, w, p.W, reinterpret_cast<int32_t*>(sm_max), L::kThreads);
        walk.init_balanced(p.seqlens, p.B, p.S, w, p.W, st);
    } else {
        const int unit = pair / p.row_blocks;
        walk.init_fixed(p.seqlens, p.B, p.S, unit / p.S, unit % p.S);
    }
    const int rho0 = rb * 128 + (int)cta * 64;  // first (query, head) row of this CTA
    Piece pc;
    int pi = 0;  // non-empty pieces walked so far (phase of the per-piece barriers)

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer of Q and the K ring
        // (both CTAs).  Every "full" barrier lives in the leader and counts the bytes of BOTH CTAs.
        if constexpr (PG != 0) {
            constexpr int NB = 64 / PG;  // boxes per column block of this CTA's 64 rows
            const int run = lane % NB;
            const uint32_t q_full_l = mapa(smem_u32(q_full), 0);
            int ks = 0;
            uint32_t kph = 1;
            bool ok = true;
            while (ok && walk.next(pc)) {
                if (pc.n_tiles == 0) continue;
                const int32_t T = p.seqlens[pc.b];
                if (pi > 0 && !(ok = __all_sync(0xffffffffu, mbar_wait(q_empty, (pi - 1) & 1, ab, 13)))) break;
                if (cta == 0 && lane == 0) mbar_expect_tx(q_full, 2 * L::kQBytes);
                __syncwarp();
                if (lane < 9) tma_load_2d_pair(tiles + lane * L::kBox, &tmQ, lane * 64, pc.b * p.rows_total + rho0, q_full_l);
                const uint32_t tok = pc.tok_begin + (int)cta * 64 + run * PG;  // this lane's run of rows in the first tile
                int32_t next_row = p.rows.run_row(pc.b, tok, T, p.n_rows);
                for (int kt = 0; kt < pc.n_tiles && ok; ++kt) {
                    const int32_t row = next_row;
                    if (kt + 1 < pc.n_tiles) next_row = p.rows.run_row(pc.b, tok + (kt + 1) * 128, T, p.n_rows);
#pragma unroll 1
                    for (int kg = 0; kg < 9; ++kg) {
                        if (!(ok = __all_sync(0xffffffffu, mbar_wait(&kempty[ks], kph, ab, 1)))) break;
                        if (cta == 0 && lane == 0) mbar_expect_tx(&kfull[ks], 2 * L::kKGroup);
                        __syncwarp();
                        if (lane < NB)
                            tma_load_2d_pair(tiles + L::kOffK + ks * L::kKGroup + run * PG * 128, &tmC, kg * 64, row,
                                             mapa(smem_u32(&kfull[ks]), 0));
                        if (++ks == L::kNK) { ks = 0; kph ^= 1; }
                    }
                }
                ++pi;
            }
        } else {
            const uint32_t e = elect_one();
            const uint32_t q_full_l = mapa(smem_u32(q_full), 0);
            int ks = 0;
            uint32_t kph = 1;  // parity that means "slot is free"
            bool ok = true;
            while (ok && warp_all(walk.next(pc))) {
                const int n_tiles = warp_uniform(pc.n_tiles);
                if (n_tiles == 0) continue;
                // Q rows of this piece's sequence; the previous piece's Qh Kh^T must all have completed
                if (pi > 0 && !(ok = warp_all(mbar_wait(q_empty, (pi - 1) & 1, ab, 13)))) break;
                if (cta == 0) mbar_expect_tx(q_full, 2 * L::kQBytes, e);
                const int32_t q_row = warp_uniform(pc.b * p.rows_total + rho0);
#pragma unroll
                for (int kb = 0; kb < 9; ++kb)
                    tma_load_2d_pair(tiles + kb * L::kBox, &tmQ, kb * 64, q_row, q_full_l, e);
                // K groups in the order (tile, column third); a tile never straddles a page
                int64_t tile_row = p.rows.row(pc.b, pc.tok_begin);
                for (int kt = 0; kt < n_tiles && ok; ++kt) {
                    const int32_t row = warp_uniform((int32_t)(tile_row + cta * 64));
                    // the next tile's row is fetched while this tile's slots are waited for
                    if (kt + 1 < n_tiles)
                        tile_row = p.rows.paged() ? p.rows.row(pc.b, pc.tok_begin + (kt + 1) * 128) : tile_row + 128;
#pragma unroll 1
                    for (int kg = 0; kg < 3; ++kg) {
                        if (!(ok = warp_all(mbar_wait(&kempty[ks], kph, ab, 1)))) break;
                        if (cta == 0) mbar_expect_tx(&kfull[ks], 2 * L::kKGroup, e);
                        const uint32_t bar = mapa(smem_u32(&kfull[ks]), 0);
                        uint8_t* dst = tiles + L::kOffK + ks * L::kKGroup;
#pragma unroll
                        for (int i = 0; i < 3; ++i) tma_load_2d_pair(dst + i * L::kBox, &tmC, (3 * kg + i) * 64, row, bar, e);
                        if (++ks == L::kNK) { ks = 0; kph ^= 1; }
                    }
                }
                ++pi;
            }
        }
    } else if (warp == L::kVProducerWarp) {
        // ------------------------------------------------------------------ TMA producer of the V ring (both
        // CTAs): the two rings fill independently of one another.  V groups in the order (tile, token half); a V slot is free
        // only after P.V of the previous tile, i.e. after Qh Kh^T of this tile has read the same cache rows
        // as K boxes, so the V boxes come out of L2 (with column halves, whose ring holds two tiles, V may be
        // asked for before K; then K comes out of L2).
        if constexpr (PG != 0) {
            constexpr int NB = L::kVRows / PG, NG = 128 / L::kVRows;  // boxes of a column block, groups of a tile
            const int run = lane % NB, mi = lane / NB;
            int vs = 0;
            uint32_t vph = 1;
            bool ok = true;
            while (ok && walk.next(pc)) {
                if (pc.n_tiles == 0) continue;
                const int32_t T = p.seqlens[pc.b];
                if (pi > 0 && !(ok = __all_sync(0xffffffffu, mbar_wait(epi_done, (pi - 1) & 1, ab, 16)))) break;
                const uint32_t tok = pc.tok_begin + run * PG;
                int32_t next_row = p.rows.run_row(pc.b, tok, T, p.n_rows);
                for (int vg = 0; vg < NG * pc.n_tiles; ++vg) {
                    const int32_t row = next_row;
                    const int32_t left = T - (pc.tok_begin + vg * L::kVRows);
                    const int cut = cut_run<PG>(left, L::kVRows);
                    if (vg + 1 < NG * pc.n_tiles) next_row = p.rows.run_row(pc.b, tok + (vg + 1) * L::kVRows, T, p.n_rows);
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait(&vempty[vs], vph, ab, 2)))) break;
                    if (cta == 0 && lane == 0) mbar_expect_tx(&vfull[vs], 2 * L::kVGroup);
                    __syncwarp();
                    uint8_t* dst = tiles + L::kOffV + vs * L::kVGroup;
                    const uint32_t bar = mapa(smem_u32(&vfull[vs]), 0);
                    if (mi < 4 && run != cut)
                        tma_load_2d_pair(dst + mi * L::kVBox + run * PG * 128, &tmC,
                                         256 * (mi >> 1) + 128 * (int)cta + 64 * (mi & 1), row, bar);
                    if (cut >= 0)
                        load_cut_run<PG, 4>(cut_maps, lane, left % PG, __shfl_sync(0xffffffffu, row, cut), p.n_rows,
                                            [&](const CUtensorMap* m, int b, int r, int32_t y) {
                                                tma_load_2d_pair(dst + b * L::kVBox + (cut * PG + r) * 128, m,
                                                                 256 * (b >> 1) + 128 * (int)cta + 64 * (b & 1), y, bar);
                                            });
                    if (++vs == L::kNV) { vs = 0; vph ^= 1; }
                }
                ++pi;
            }
        } else {
            const uint32_t e = elect_one();
            int vs = 0;
            uint32_t vph = 1;
            bool ok = true;
            while (ok && warp_all(walk.next(pc))) {
                const int n_tiles = warp_uniform(pc.n_tiles);
                if (n_tiles == 0) continue;
                // the V ring doubles as the output staging of the previous piece
                if (pi > 0 && !(ok = warp_all(mbar_wait(epi_done, (pi - 1) & 1, ab, 16)))) break;
                int64_t tile_row = p.rows.row(pc.b, pc.tok_begin);
                for (int vt = 0; vt < n_tiles && ok; ++vt) {
                    const int64_t row0 = tile_row;
                    if (vt + 1 < n_tiles)
                        tile_row = p.rows.paged() ? p.rows.row(pc.b, pc.tok_begin + (vt + 1) * 128) : tile_row + 128;
#pragma unroll 1
                    for (int vh = 0; vh < 2; ++vh) {
                        if (!(ok = warp_all(mbar_wait(&vempty[vs], vph, ab, 2)))) break;
                        if (cta == 0) mbar_expect_tx(&vfull[vs], 2 * L::kVGroup, e);
                        const int32_t row = warp_uniform((int32_t)(row0 + vh * 64));
                        const uint32_t bar = mapa(smem_u32(&vfull[vs]), 0);
                        uint8_t* dst = tiles + L::kOffV + vs * L::kVGroup;
                        // box (m, i): latent columns [256m + 128cta + 64i, +64) -- this CTA's half of MMA m's N
#pragma unroll
                        for (int mi = 0; mi < 2 * L::kBlocks; ++mi)
                            tma_load_2d_pair(dst + mi * L::kBox, &tmC, 256 * (blk0 + (mi >> 1)) + 128 * (int)cta + 64 * (mi & 1),
                                             row, bar, e);
                        if (++vs == L::kNV) { vs = 0; vph ^= 1; }
                    }
                }
                ++pi;
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leader CTA only)
        if (cta == 0) {
            const uint32_t e = elect_one();
            constexpr uint32_t idesc_qk = idesc_bf16(128, 128, 0, 0);
            constexpr uint32_t idesc_pv = idesc_bf16(128, 256, 0, 1);
            const uint64_t q_desc = desc_kmajor_sw128(smem_u32(tiles));
            const uint64_t p_desc = desc_kmajor_sw128(smem_u32(tiles + L::kOffP));
            int ks = 0, vs = 0;
            uint32_t kph = 0, vph = 0;
            int gt = 0;  // tiles issued so far: score buffer = gt & 1, phase = (gt >> 1) & 1
            auto issue_qk = [&](int n) -> bool {
                const uint32_t d = tmem_base + kAColS + (uint32_t)(n & 1) * 64;
#pragma unroll 1
                for (int g = 0; g < 9 / L::kKBlocks; ++g) {
                    if (!warp_all(mbar_wait_fast(&kfull[ks], kph, ab, 3))) return false;
                    tc_fence_after();
                    // descriptors as low words: the high word is a constant, stepping is one 32-bit add
                    const uint32_t kd = desc_lo(desc_kmajor_sw128(smem_u32(tiles + L::kOffK + ks * L::kKGroup)));
                    const uint32_t qd = desc_lo(q_desc) + ((g * L::kKBlocks * L::kBox) >> 4);
                    if (g == 0)
                        umma_ss2_lo<false>(d, qd, kd, idesc_qk, e);  // the tile's first MMA overwrites S
                    else
                        umma_ss2_lo<true>(d, qd, kd, idesc_qk, e);
#pragma unroll
                    for (int i = 0; i < L::kKBlocks; ++i)
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            if ((i | kk) != 0)
                                umma_ss2_lo<true>(d, qd + ((i * L::kBox + kk * 32) >> 4), kd + ((i * L::kBox + kk * 32) >> 4),
                                                  idesc_qk, e);
                    umma_commit2(&kempty[ks], 3, e);
                    if (++ks == L::kNK) { ks = 0; kph ^= 1; }
                }
                umma_commit2(&s_full[n & 1], 3, e);
                return true;
            };
            bool ok = true;
            while (ok && warp_all(walk.next(pc))) {
                const int n_tiles = warp_uniform(pc.n_tiles);
                if (n_tiles == 0) continue;
                if (!(ok = warp_all(mbar_wait(q_full, pi & 1, ab, 4)))) break;
                tc_fence_after();
                if (!(ok = issue_qk(gt))) break;
                for (int t = 0; t < n_tiles && ok; ++t) {
                    const int n = gt + t;
                    if (t + 1 < n_tiles) {
                        if (!(ok = issue_qk(n + 1))) break;
                    } else {
                        umma_commit2(q_empty, 3, e);  // every Qh Kh^T of this piece has been issued
                    }
                    if (!(ok = warp_all(mbar_wait_fast(&p_ready[n & 1], (n >> 1) & 1, ab, 5)))) break;
                    // the first P.V of a piece overwrites O: the previous piece's O must have been read
                    if (t == 0 && pi > 0 && !(ok = warp_all(mbar_wait(o_free, (pi - 1) & 1, ab, 14)))) break;
                    tc_fence_after();
#pragma unroll 1
                    for (int g = 0; g < 128 / L::kVRows; ++g) {
                        if (!(ok = warp_all(mbar_wait_fast(&vfull[vs], vph, ab, 6)))) break;
                        tc_fence_after();
                        const uint32_t vd = desc_lo(desc_mnmajor_sw128(smem_u32(tiles + L::kOffV + vs * L::kVGroup), L::kVBox));
                        const int tok = g * L::kVRows;  // P: 64 tokens a k-block
                        const uint32_t pd = desc_lo(p_desc) + ((tok / 64 * L::kBox + tok % 64 * 2) >> 4);
#pragma unroll
                        for (int m = 0; m < L::kBlocks; ++m) {
                            const uint32_t dm = tmem_base + kAColO + (uint32_t)m * 128;
                            const uint32_t vm = vd + ((m * 2 * L::kVBox) >> 4);
                            if ((t | g) == 0)
                                umma_ss2_lo<false>(dm, pd, vm, idesc_pv, e);  // first P.V of a piece
                            else
                                umma_ss2_lo<true>(dm, pd, vm, idesc_pv, e);
#pragma unroll
                            for (int kk = 1; kk < L::kVRows / 16; ++kk)
                                umma_ss2_lo<true>(dm, pd + ((kk * 32) >> 4), vm + ((kk * 2048) >> 4), idesc_pv, e);
#pragma unroll
                            for (int n = 1; n < L::kPTerms; ++n)  // the other terms of P
#pragma unroll
                                for (int kk = 0; kk < L::kVRows / 16; ++kk) {
                                    const uint32_t d = m == 0 ? tmem_base + kAColRest : dm;
                                    const uint32_t a = pd + ((n * L::kPTerm + kk * 32) >> 4), b = vm + ((kk * 2048) >> 4);
                                    if (m == 0 && n == 1 && kk == 0 && (t | g) == 0)
                                        umma_ss2_lo<false>(d, a, b, idesc_pv, e);
                                    else
                                        umma_ss2_lo<true>(d, a, b, idesc_pv, e);
                                }
                        }
                        umma_commit2(&vempty[vs], 3, e);
                        if (++vs == L::kNV) { vs = 0; vph ^= 1; }
                    }
                    if (ok) umma_commit2(&pv_done[n & 1], 3, e);
                }
                gt += n_tiles;
                ++pi;
            }
        }
    } else {
        // ------------------------------------------------------------------ softmax
        const int q = warp & 3;              // TMEM lane quadrant this warp may access
        const int ch = (warp - 2) >> 2;      // which 32 of the lane's 64 score columns
        const int Lr = q * 32 + lane;        // TMEM lane
        const int r = Lr & 63;               // row within this CTA
        const int hf = Lr >> 6;              // token half of each 128-token tile / column half of each O block
        const int part = hf * 2 + ch;        // one of the four threads of row r
        const int rho = rho0 + r;            // (query, head) row of the sequence
        const bool row_valid = rho < p.rows_total;
        const int pq = row_valid ? rho / p.h_q : 0;
        const uint32_t lane_base = tmem_base + ((uint32_t)(q * 32) << 16);
        const uint32_t p_ready_l[2] = {mapa(smem_u32(&p_ready[0]), 0), mapa(smem_u32(&p_ready[1]), 0)};
        const uint32_t o_free_l = mapa(smem_u32(o_free), 0);
        int gt = 0;  // tiles walked so far
        int ec = 0;  // completed phases of the `epi` barrier

        while (walk.next(pc)) {
            GQLA_DEBUG_CHECK(pc.b >= 0 && pc.b < p.B, p.status, 32);  // a piece names a sequence of the batch
            const int32_t T = p.seqlens[pc.b];
            const int64_t slot0 = (int64_t)pc.b * p.S;
            GQLA_DEBUG_CHECK(pc.n_tiles == 0 || (pc.k >= 0 && pc.k < p.S), p.status, 33);  // ... and one of its S slots
            GQLA_DEBUG_CHECK(pc.tok_begin >= 0 && pc.tok_begin <= pc.tok_end && pc.tok_end <= (T > 0 ? T : 0), p.status, 34);
            GQLA_DEBUG_CHECK(pc.n_tiles == (pc.tok_end > pc.tok_begin ? (pc.tok_end - pc.tok_begin + 127) / 128 : 0), p.status, 35);
            GQLA_DEBUG_CHECK(!p.balanced || pc.tok_begin % 128 == 0, p.status, 36);  // balanced pieces start on tile boundaries
            GQLA_DEBUG_CHECK(pc.fill_begin >= 0 && pc.fill_begin <= pc.fill_end && pc.fill_end <= p.S || pc.fill_end == 0, p.status, 37);
            // split slots this worker marks empty
            if (part == 0 && blk0 == 0 && row_valid && p.lse_part != nullptr)
                for (int kk = pc.fill_begin; kk < pc.fill_end; ++kk) p.lse_part[(slot0 + kk) * p.rows_total + rho] = -INFINITY;
            if (pc.n_tiles == 0 && p.balanced) continue;  // an empty sequence: its slots were marked above
            int32_t lim = visible_limit(T, p.s_q, pq);
            if (lim > pc.tok_end) lim = pc.tok_end;
            lim -= pc.tok_begin;
            if (!row_valid) lim = 0;
            float m_used = -INFINITY, l = 0.f;
            bool ok = true;

            for (int t = 0; t < pc.n_tiles && ok; ++t) {
                const int n = gt + t;
                const int sb = n & 1;
                const uint32_t nph = (n >> 1) & 1;
                ok = __all_sync(0xffffffffu, mbar_wait(&s_full[sb], nph, ab, 7));
                if (!ok) break;
                tc_fence_after();
                const int tok0 = t * 128 + hf * 64 + ch * 32;
                uint32_t x[32];
                tmem_ld32(lane_base + kAColS + (uint32_t)sb * 64 + ch * 32, x);
                tmem_wait_ld();
                const bool full = tok0 + 32 <= lim;  // every score of this thread is visible
                float mx = -INFINITY;
                if (full) {
#pragma unroll
                    for (int c = 0; c < 32; ++c) mx = fmaxf(mx, __uint_as_float(x[c]));
                } else {
#pragma unroll
                    for (int c = 0; c < 32; ++c)
                        if (tok0 + c < lim) mx = fmaxf(mx, __uint_as_float(x[c]));
                }
                // the other three parts of this row live in other warps
                float* mxs = sm_max + sb * 256;
                mxs[part * 64 + r] = mx;
                __syncwarp();
                if (lane == 0) mbar_arrive(&xch[sb]);
                ok = __all_sync(0xffffffffu, mbar_wait(&xch[sb], nph, ab, 10));
                if (!ok) break;
                mx = fmaxf(fmaxf(mxs[r], mxs[64 + r]), fmaxf(mxs[128 + r], mxs[192 + r]));
                const float m_t = mx * p.scale_log2;
                const bool need = m_t > m_used + 8.0f;
                const float factor = need ? ex2(m_used - m_t) : 1.f;
                if (need) {
                    l *= factor;
                    m_used = m_t;
                }
                const float m_sub = m_used == -INFINITY ? 0.f : m_used;
                uint32_t pk[16 * L::kPTerms];  // [term][pair of columns]
                if (full) {
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        const float e0 = ex2(fmaf(__uint_as_float(x[c]), p.scale_log2, -m_sub));
                        const float e1 = ex2(fmaf(__uint_as_float(x[c + 1]), p.scale_log2, -m_sub));
                        l += e0 + e1;
                        split_bf16<L::kPTerms>(e0, e1, pk + c / 2, 16);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        const float e0 = tok0 + c < lim ? ex2(fmaf(__uint_as_float(x[c]), p.scale_log2, -m_sub)) : 0.f;
                        const float e1 =
                            tok0 + c + 1 < lim ? ex2(fmaf(__uint_as_float(x[c + 1]), p.scale_log2, -m_sub)) : 0.f;
                        l += e0 + e1;
                        split_bf16<L::kPTerms>(e0, e1, pk + c / 2, 16);
                    }
                }
                // O may be rescaled, and the P buffer rewritten, only once P.V(n-1) has completed
                if (t > 0) {
                    ok = __all_sync(0xffffffffu, mbar_wait(&pv_done[(n - 1) & 1], ((n - 1) >> 1) & 1, ab, 8));
                    if (!ok) break;
                    tc_fence_after();
                }
                if (__any_sync(0xffffffffu, need) && t > 0) {
                    // this thread's share of the lane's O: columns [128m + 64ch, +64) for m = 0, 1
#pragma unroll 1
                    for (int c = 0; c < (L::kPTerms > 1 ? 6 : 2 * L::kBlocks); ++c) {
                        const uint32_t col = (c < 4 ? kAColO + (uint32_t)(c >> 1) * 128 : kAColRest) + ch * 64 + (c & 1) * 32;
                        uint32_t o[32];
                        tmem_ld32(lane_base + col, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * factor);
                        tmem_st32(lane_base + col, o);
                    }
                    tmem_wait_st();
                }
                // P row r, k-block hf: 128 bytes = 8 chunks of 8 bf16, chunk index XORed with (r & 7)
                uint8_t* prow = tiles + L::kOffP + hf * L::kBox + r * 128;
#pragma unroll
                for (int c4 = 0; c4 < 4 * L::kPTerms; ++c4)
                    *reinterpret_cast<uint4*>(prow + (c4 >> 2) * L::kPTerm + (((ch * 4 + (c4 & 3)) ^ (r & 7)) << 4)) =
                        make_uint4(pk[4 * c4], pk[4 * c4 + 1], pk[4 * c4 + 2], pk[4 * c4 + 3]);
                fence_proxy_async_smem();  // generic-proxy writes of P -> visible to the tensor core
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(p_ready_l[sb]);
            }

            // -------------------------------------------------------------- epilogue: normalise and store
            const int n_last = gt + pc.n_tiles - 1;
            if (pc.n_tiles > 0 && ok)
                ok = __all_sync(0xffffffffu, mbar_wait(&pv_done[n_last & 1], (n_last >> 1) & 1, ab, 9));
            tc_fence_after();
            sm_l[part * 64 + r] = l;
            __syncwarp();
            if (lane == 0) mbar_arrive(fin);
            if (!__all_sync(0xffffffffu, mbar_wait(fin, pi & 1, ab, 11))) ok = false;
            const float Lt = (sm_l[r] + sm_l[64 + r]) + (sm_l[128 + r] + sm_l[192 + r]);
            const bool live = ok && pc.n_tiles > 0 && Lt > 0.f && m_used > -INFINITY;
            const float inv = live ? 1.f / Lt : 0.f;
            // The CTA's 64 output rows leave through shared memory (P and the V ring are idle now: the last
            // P.V has completed) as bulk stores.  The padded pitches keep the 16-byte stores of a quarter warp on
            // distinct banks.
            uint8_t* stage = tiles + L::kOffP;
            if constexpr (FINAL) {
                // whole-sequence call: the final bf16 rows (1 KB each) fit the staging at once -- one pass
                uint4* dst = reinterpret_cast<uint4*>(stage + r * L::kOutPitch + (128 * hf + 64 * ch) * 2);
#pragma unroll 1
                for (int mc = 0; mc < 2 * L::kBlocks; ++mc) {  // (m, 32-column half) of this thread's 64 columns of each m
                    const int m = mc >> 1, c = (mc & 1) * 32;
                    uint32_t o[32];
                    if (pc.n_tiles > 0 && ok) {  // warp-uniform
                        tmem_ld32(lane_base + kAColO + m * 128 + ch * 64 + c, o);
                        tmem_wait_ld();
                    }
                    auto pk = [&](int e) -> uint32_t {  // columns e, e + 1 of this chunk, normalised (0 for a dead row)
                        return live ? pack_bf16(__uint_as_float(o[e]) * inv, __uint_as_float(o[e + 1]) * inv) : 0u;
                    };
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        dst[(256 * m + c) * 2 / 16 + i] = make_uint4(pk(8 * i), pk(8 * i + 2), pk(8 * i + 4), pk(8 * i + 6));
                }
                fence_proxy_async_smem();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(o_free_l);
                if (lane == 0) mbar_arrive(epi);
                if (!__all_sync(0xffffffffu, mbar_wait(epi, ec & 1, ab, 12))) ok = false;
                ++ec;
                if (ok && lane < 8) {
                    const int rr = (warp - 2) * 8 + lane;
                    if (rho0 + rr < p.rows_total) {
                        bulk_store(p.o_final + ((int64_t)pc.b * p.rows_total + rho0 + rr) * 512 + 256 * blk0,
                                   stage + rr * L::kOutPitch, L::kBlocks * 256 * 2);
                        bulk_commit();
                        bulk_wait_read();
                    }
                }
            } else {
                // fp32 partials: every warp stages and ships 32 rows x 64 columns of MMA m's block by itself (256-byte
                // bulk stores, one per row), the block of m = 1 behind that of m = 0.  No warp waits for another, so one
                // stages while others' stores drain (73 sequences of 300-500 rows: 53.6 us a step with two passes of the whole
                // CTA and 1 KB stores, 52.3 like this; straight from registers 54.9; an SM writes about 30 B per clock).
                uint8_t* own = stage + ((warp - 2) * 32 + lane) * L::kWarpPitch;
                float* grow = p.o_part + ((slot0 + pc.k) * p.rows_total + rho) * 512 + 256 * blk0 + 128 * hf + 64 * ch;
#pragma unroll 1
                for (int m = 0; m < L::kBlocks; ++m) {
                    if (m == 1) bulk_wait_read();  // this lane's row of m = 0 has left the staging
#pragma unroll 1
                    for (int c = 0; c < 64; c += 32) {
                        uint32_t o[32];
                        if (pc.n_tiles > 0 && ok) {  // warp-uniform
                            tmem_ld32(lane_base + kAColO + m * 128 + ch * 64 + c, o);
                            tmem_wait_ld();
                            if (L::kPTerms > 1 && m == 0) {
                                uint32_t rest[32];
                                tmem_ld32(lane_base + kAColRest + ch * 64 + c, rest);
                                tmem_wait_ld();
#pragma unroll
                                for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) + __uint_as_float(rest[i]));
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            reinterpret_cast<float4*>(own)[c / 4 + i] =
                                live ? make_float4(__uint_as_float(o[4 * i]) * inv, __uint_as_float(o[4 * i + 1]) * inv,
                                                   __uint_as_float(o[4 * i + 2]) * inv, __uint_as_float(o[4 * i + 3]) * inv)
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    if (m == L::kBlocks - 1) {  // O has been read: the next piece's first P.V may overwrite it
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(o_free_l);
                    }
                    fence_proxy_async_smem();  // staged row -> visible to the bulk-copy engine
                    if (row_valid && ok) bulk_store(grow + 256 * m, own, 256);
                    bulk_commit();
                    __syncwarp();
                }
                bulk_wait_read();
            }
            // staging (and with it P and the V ring) is free again once every warp's stores have read it
            __syncwarp();
            if (lane == 0) mbar_arrive(epi_done);
            if (!__all_sync(0xffffffffu, mbar_wait(epi_done, pi & 1, ab, 12))) ok = false;
            if (row_valid && part == 0 && blk0 == 0 && p.lse_part != nullptr)
                p.lse_part[(slot0 + pc.k) * p.rows_total + rho] =
                    live ? (m_used + log2f(Lt)) * 0.6931471805599453f : -INFINITY;
            gt += pc.n_tiles;
            ++pi;
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // neither CTA leaves while the other may still signal its barriers
    if (warp == 1) tmem_dealloc2(tmem_base, 512);
}

}  // namespace tc
}  // namespace gqla
