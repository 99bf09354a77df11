// One-shot cache expansion on CTA pairs (Sec. 3.1: k^C = W^UK c, v^C = W^UV c per group):
//   [K_C | V][n, :] = c[n, 0:r_kv] . [W^UK ; W^UV]      a plain GEMM  N x r_kv x (2 g d_h).
// Persistent CTA pairs walk units of 256 cache rows (128 per CTA) x `unit_tiles` column tiles.  A unit's latent rows are
// loaded ONCE and stay in shared memory while the pair walks its column tiles (all 2 g d_h / 256 of them when there are
// rows enough); the weights stream through a ring, each CTA fetching half of every B tile (cta_group::2 MMAs of
// 256 x 256 x 16 read B from both CTAs), so the weights cross L2 -> SM once per 256 rows instead of once per 128.
// A k-block of the latent rows is free again as soon as the last column tile's MMAs have read it, and the next unit's
// rows are loaded into it right away: with two 256-column accumulators in TMEM the epilogue warps store tile t while
// the MMAs of tile t + 1 run, across units too, and the tensor core only waits at the very first unit of a pair.
// (One pair per 256 rows and launch slot, as this kernel was before, paid set-up, the load of the rows and the last
// tile's store once per unit: 452 us against 413 us on 224 672 rows back to back at the power cap, 61 against 48 us on
// 20 000.)  The output leaves through
// swizzled shared-memory staging boxes and TMA stores, 64 columns x 32 rows at a time: one thread per row
// writing its row straight to global memory costs more store instructions than the MMAs give it time for.  Every
// epilogue warp has a box of its own: with one box of 128 rows the four warps met at two barriers per 64 columns and
// waited together for its store (the two in turn on one GPU: 224 672 rows 430 against 428 us, 20 000 rows 49.1 against 48.3;
// GPUs differ by more).
// Warp roles per CTA: warp 0 TMA producer, warp 1 TMEM owner (+ MMA issuer in the leader), warps 2-5
// epilogue (TMEM lane = row).
#pragma once
#include "tc_common.cuh"


namespace gqla {
namespace tc {

struct ExpandParams {
    int64_t n_rows;          // cache rows N
    int32_t row_blocks;      // ceil(N / 256)
    int32_t unit_tiles;      // column tiles of a unit (divides the 2 g d_h / 256 tiles of a row block)
    int32_t g, r_kv, d_r;    // d_h = 128
    void* k_c;               // [N, g, 128]
    void* v;                 // [N, g, 128]
    const void* cache;       // for the k_R copy
    void* k_r;               // [N, d_r] or null
    int64_t cache_stride;    // elements
    int32_t* status;
};

struct ExpandSmem {
    static constexpr int kKBlocks = 8;                   // r_kv = 512
    static constexpr int kABytes = kKBlocks * 16384;     // 128 rows x 512, eight 64-wide k-blocks
    static constexpr int kBStage = 2 * 8192;             // 64 k x 128 n: this CTA's half of a 256-column tile
    // ring of B stages: measured on the C2 cache, 4 stages 0.498 ms, 5 stages 0.464 ms (the weights come out of
    // L2 and every k-block is only 512 cycles of tensor work)
    static constexpr int kStages = 5;
    static constexpr int kOutBytes = 16384;              // output staging: a box of 32 rows x 64 bf16 per epilogue warp, 128-byte swizzle
    static constexpr int kTileBytes = kABytes + kStages * kBStage + kOutBytes;
    // a_full[kKBlocks], a_empty[kKBlocks], b_full[], b_empty[], acc_full[2], acc_empty[2]
    static constexpr int kNumBars = 2 * kKBlocks + 2 * kStages + 4;
    static constexpr int kThreads = 192;
    static constexpr int kTotal = 1024 + kTileBytes + kNumBars * 8 + 16;
    static_assert(kTotal <= 232448, "shared memory budget of one CTA");
    static_assert(OneCtaPerSM<kTotal>::value, "");
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(ExpandSmem::kThreads, 1)
expand_tc_kernel(const ExpandParams p, const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmK,
                 const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmOK,
                 const __grid_constant__ CUtensorMap tmOV) {
    using L = ExpandSmem;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* a_smem = tiles;
    uint8_t* b_smem = tiles + L::kABytes;
    uint8_t* out_smem = b_smem + L::kStages * L::kBStage;
    uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + L::kTileBytes);
    uint64_t* a_full = bars;                       // [kKBlocks] leader: both CTAs' latent rows have landed
    uint64_t* a_empty = a_full + L::kKBlocks;      // [kKBlocks] per CTA: the unit's last tile has read the k-block
    uint64_t* b_full = a_empty + L::kKBlocks;      // [kStages] leader: both halves of a B stage have landed
    uint64_t* b_empty = b_full + L::kStages;       // [kStages] per CTA
    uint64_t* acc_full = b_empty + L::kStages;     // [2] per CTA (multicast commit)
    uint64_t* acc_empty = acc_full + 2;            // [2] leader: the epilogue warps of both CTAs have read the tile
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + L::kNumBars);
    volatile int32_t* abort_flag = reinterpret_cast<volatile int32_t*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t cta = cluster_ctarank();
    const Abort ab{abort_flag, p.status};
    const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const int col_units = p.g / p.unit_tiles;        // a row block has g column tiles of 256 (K_C first, then V)
    const int n_units = p.row_blocks * col_units;    // unit u: row block u / col_units, tiles [(u % col_units) * unit_tiles, ..)
    auto row_of = [&](int u) -> int64_t { return (int64_t)(u / col_units) * 256 + cta * 128; };  // first row of this CTA

    if (threadIdx.x == 0) {
        for (int i = 0; i < L::kNumBars; ++i) mbar_init(&bars[i], (&bars[i] == &acc_empty[0] || &bars[i] == &acc_empty[1]) ? 8 : 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc2(tmem_slot, 512);
        tmem_relinquish2();
    }
    pdl_launch_dependents();
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer (both CTAs)
        if (elect_one()) {
            tma_prefetch_desc(&tmA);
            tma_prefetch_desc(&tmK);
            tma_prefetch_desc(&tmV);
            int s = 0;
            uint32_t ph = 1, aph = 1;  // parities that mean "free"
            bool ok = true;
            for (int u = pair; u < n_units && ok; u += n_pairs, aph ^= 1) {
                const int32_t row = (int32_t)row_of(u);
                const int t0 = (u % col_units) * p.unit_tiles;
                for (int t = t0; t < t0 + p.unit_tiles && ok; ++t) {
                    // this CTA supplies columns [128 cta, +128) of the tile: one whole group of one plane
                    const int jj = (2 * t) % p.g + (int)cta;
                    const CUtensorMap* tmB = 2 * t >= p.g ? &tmV : &tmK;
                    for (int kb = 0; kb < L::kKBlocks; ++kb) {
                        if (t == t0) {  // a unit's latent rows arrive with its first tile, k-block by k-block
                            if (!(ok = mbar_wait(&a_empty[kb], aph, ab, 6))) break;
                            if (cta == 0) mbar_expect_tx(&a_full[kb], 2 * 16384);
                            tma_load_2d_pair(a_smem + kb * 16384, &tmA, kb * 64, row, mapa(smem_u32(&a_full[kb]), 0));
                        }
                        if (!(ok = mbar_wait(&b_empty[s], ph, ab, 1))) break;
                        if (cta == 0) mbar_expect_tx(&b_full[s], 2 * L::kBStage);
                        const uint32_t bar = mapa(smem_u32(&b_full[s]), 0);
                        uint8_t* dst = b_smem + s * L::kBStage;
                        tma_load_2d_pair(dst, tmB, 0, jj * p.r_kv + kb * 64, bar);
                        tma_load_2d_pair(dst + 8192, tmB, 64, jj * p.r_kv + kb * 64, bar);
                        if (++s == L::kStages) { s = 0; ph ^= 1; }
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leader CTA only)
        if (cta == 0 && elect_one()) {
            constexpr uint32_t idesc = idesc_bf16(256, 256, 0, 1);
            const uint32_t a_lo = desc_lo(desc_kmajor_sw128(smem_u32(a_smem)));
            int s = 0;
            uint32_t ph = 0;
            uint32_t aph = 0;
            bool ok = true;
            int at = 0;  // tiles issued so far: accumulator at & 1, phase (at >> 1) & 1
            for (int u = pair; u < n_units && ok; u += n_pairs, aph ^= 1) {
                for (int t = 0; t < p.unit_tiles && ok; ++t, ++at) {
                    const int buf = at & 1;
                    const bool first = t == 0, last = t + 1 == p.unit_tiles;
                    if (!(ok = mbar_wait(&acc_empty[buf], ((at >> 1) & 1) ^ 1, ab, 3))) break;
                    tc_fence_after();
                    const uint32_t d = tmem_base + (uint32_t)buf * 256;
                    for (int kb = 0; kb < L::kKBlocks; ++kb) {
                        if (first && !(ok = mbar_wait(&a_full[kb], aph, ab, 2))) break;
                        if (!(ok = mbar_wait(&b_full[s], ph, ab, 4))) break;
                        tc_fence_after();
                        const uint32_t b_lo = desc_lo(desc_mnmajor_sw128(smem_u32(b_smem + s * L::kBStage), 8192));
                        if (kb == 0)
                            umma_ss2_lo<false>(d, a_lo, b_lo, idesc);
                        else
                            umma_ss2_lo<true>(d, a_lo + ((kb * 16384) >> 4), b_lo, idesc);
#pragma unroll
                        for (int ks = 1; ks < 4; ++ks)
                            umma_ss2_lo<true>(d, a_lo + ((kb * 16384 + ks * 32) >> 4), b_lo + ((ks * 2048) >> 4), idesc);
                        umma_commit2(&b_empty[s], 3);
                        if (last) umma_commit2(&a_empty[kb], 3);
                        if (++s == L::kStages) { s = 0; ph ^= 1; }
                    }
                    if (ok) umma_commit2(&acc_full[buf], 3);
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue: TMEM lane = row
        const int q = warp & 3;
        const uint32_t acc_empty_l[2] = {mapa(smem_u32(&acc_empty[0]), 0), mapa(smem_u32(&acc_empty[1]), 0)};
        uint8_t* box = out_smem + q * 4096;  // this warp's 32 rows x 64 columns
        bool ok = true;
        int at = 0;
        for (int u = pair; u < n_units && ok; u += n_pairs) {
            const int64_t warp_row = row_of(u) + q * 32, n = warp_row + lane;
            const int t0 = (u % col_units) * p.unit_tiles;
            if (t0 == 0 && n < p.n_rows && p.k_r != nullptr) {  // k^R is carried over unchanged
                const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.cache) +
                                                                  n * p.cache_stride + p.r_kv);
                uint4* kr = reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.k_r) + n * p.d_r);
                for (int c = 0; c < p.d_r / 8; ++c) kr[c] = src[c];
            }
            for (int t = t0; t < t0 + p.unit_tiles && ok; ++t, ++at) {
                const int buf = at & 1;
                ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (at >> 1) & 1, ab, 5));
                if (!ok) break;
                tc_fence_after();
                const CUtensorMap* tmO = 2 * t >= p.g ? &tmOV : &tmOK;
                const int col_base = ((2 * t) % p.g) * 128;  // first column of the tile in its plane's [N, g * 128] rows
#pragma unroll 1
                for (int cb = 0; cb < 4; ++cb) {
                    uint32_t v[64];
                    tmem_ld32(tmem_addr(tmem_base, q * 32, buf * 256 + cb * 64), v);
                    tmem_ld32(tmem_addr(tmem_base, q * 32, buf * 256 + cb * 64 + 32), v + 32);
                    tmem_wait_ld();
                    // the warp's staging box is rewritten: its last store must have finished reading
                    if (lane == 0) bulk_wait_read();
                    __syncwarp();
#pragma unroll
                    for (int c = 0; c < 8; ++c) {  // 8 chunks of 8 bf16; chunk index XORed with (row & 7)
                        uint4 o;
                        o.x = pack_bf16(__uint_as_float(v[8 * c + 0]), __uint_as_float(v[8 * c + 1]));
                        o.y = pack_bf16(__uint_as_float(v[8 * c + 2]), __uint_as_float(v[8 * c + 3]));
                        o.z = pack_bf16(__uint_as_float(v[8 * c + 4]), __uint_as_float(v[8 * c + 5]));
                        o.w = pack_bf16(__uint_as_float(v[8 * c + 6]), __uint_as_float(v[8 * c + 7]));
                        *reinterpret_cast<uint4*>(box + lane * 128 + ((c ^ (lane & 7)) << 4)) = o;
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0 && warp_row < p.n_rows) {  // a warp wholly behind the last row stores nothing
                        tma_store_2d(tmO, box, col_base + cb * 64, (int32_t)warp_row);
                        bulk_commit();
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(acc_empty_l[buf]);
            }
        }
        if (lane == 0) bulk_wait_read();  // the last store still reads the staging box
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    if (warp == 1) tmem_dealloc2(tmem_base, 512);
}

}  // namespace tc
}  // namespace gqla
