// Split merge fused with the latent up-projection (Eq. (mqa), line 6, applied to the log-sum-exp merge
// of the split partials):   o_i = W^UV_{j(i)} ( sum_k w_k o_hat_{i,k} ),  w_k = exp(lse_k - M) / sum exp.
// The merged latent output never goes to HBM: sixteen builder warps read the fp32 partials (512 contiguous
// bytes per load), weight and sum them, and write the bf16 A operand straight into shared memory in the
// 128-byte-swizzled K-major layout; warp 0 fetches W^UV[j] with TMA, warp 1 issues tcgen05.mma into a TMEM
// accumulator; the builder warps then store the 64 x 128 output tile, 32 columns each.  Both operands are
// resident in full (r_kv <= 512).
// One CTA serves one group (W^UV[j] is fetched once) and a run of its (position, head) rows, in tiles of up to 64 rows
// (M = 64 MMAs: accumulator row m sits in TMEM lane (m % 16) + 32 (m / 16)); K = r_kv in chunks of 128.  The groups' rows
// are cut into as many runs as the GPU has SMs for a group, so every SM pulls the same share of the partials: with one
// CTA per 64 rows, 192 tiles were two waves on 148 SMs and 64 tiles left half of them idle.
// The loads of a row's partials are round trips to HBM, so what counts is how few of them follow one another: the tile's
// rows are dealt to the sixteen builder warps one by one, the weights of all slots are known (eight lanes per row)
// before the first load, empty slots are passed over, and three live slots of a row are in flight together.
// Partials from HBM, kernel alone: 4 sequences of 128 heads in four slots 6.2 us (9.0 with one CTA per 64 rows and two rows
// of a warp at a time), 48 x 2 positions in three slots 21.4 (25.1), 128 sequences of 32 heads 10.1 (11.7).  The 18 warps leave
// 96 registers a thread, into which three slots of a row just fit (16 bytes of spills).  Weights and MMAs issued by converged warps
// (tc_common.cuh): one sequence of 777 rows (eight slots) 7.2 -> 6.5 us, 48 x 2 positions 17.8 -> 16.2, back to back.
#pragma once
#include "tc_common.cuh"

namespace gqla {
namespace tc {

struct CombineUpParams {
    int32_t S, s_q, h_q, g, hpg, r_kv;
    int32_t hpb;            // heads per group padded to a power of two (head slots of a position)
    int64_t positions;      // B * s_q
    int32_t run;            // rows (positions x head slots of a group) per CTA
    const float* o_part;    // [B, S, s_q*h_q, r_kv]
    const float* lse_part;  // [B, S, s_q*h_q]
    void* out;              // [B, s_q, h_q, 128] bf16
    float* lse;             // [B, s_q, h_q] or null
    int32_t* status;
};

struct CombineUpSmem {
    static constexpr int kChunkK = 128;
    static constexpr int kRows = 64;
    static constexpr int kABytes = 2 * 8192;    // 64 rows x 128 k, two 64-wide k-blocks
    static constexpr int kBBytes = 4 * 8192;    // 128 k x 128 n: (k-block, n-block) boxes of 64 x 64
    static constexpr int kMaxChunks = 4;        // r_kv <= 512: the whole A and B operands are resident at once
    static constexpr int kTileBytes = kMaxChunks * (kABytes + kBBytes);
    static constexpr int kNumBars = 3;          // a_ready b_full acc_full
    static constexpr int kBuilders = 16;        // builder warps: four rows each
    static constexpr int kThreads = 64 + 32 * kBuilders;
    static constexpr int kMaxS = 64;            // split slots the kernel takes (their weights are staged per row)
    static constexpr int kTotal = 1024 + kTileBytes + kNumBars * 8 + 16 + kRows * kMaxS * 4;
    static_assert(OneCtaPerSM<kTotal>::value, "");
};

// Read once: do not keep in L1.  A coherent load, not the read-only one: the kernel in front still writes the partials when this
// one has been launched (6.9 us at five slots of 8 sequences with either).
__device__ __forceinline__ float4 ld_partial4(const float* p) {
    float4 v;
    asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

__global__ void __launch_bounds__(CombineUpSmem::kThreads, 1)
combine_up_tc_kernel(const CombineUpParams p, const __grid_constant__ CUtensorMap tmB) {
    using L = CombineUpSmem;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* a_smem = tiles;
    uint8_t* b_smem = tiles + L::kMaxChunks * L::kABytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + L::kTileBytes);
    uint64_t* a_ready = bars;       // the builder warps have written A
    uint64_t* b_full = bars + 1;
    uint64_t* acc_full = bars + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + L::kNumBars);
    volatile int32_t* abort_flag = reinterpret_cast<volatile int32_t*>(tmem_slot + 1);
    float* sm_w = reinterpret_cast<float*>(tmem_slot + 4);  // [64][kMaxS] normalised weight of every slot of every tile row

    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const Abort ab{abort_flag, p.status};
    const int j = blockIdx.y;
    const int64_t row0 = (int64_t)blockIdx.x * p.run, group_rows = p.positions * p.hpb;
    const int n_rows = (int)(group_rows - row0 < p.run ? group_rows - row0 : p.run);  // this CTA's run, at least 1
    const int n_tiles = (n_rows + L::kRows - 1) / L::kRows;
    const int n_chunks = p.r_kv / L::kChunkK;
    const int rows_per_seq = p.s_q * p.h_q;
    pdl_launch_dependents();

    if (threadIdx.x == 0) {
        for (int i = 0; i < L::kNumBars; ++i) mbar_init(&bars[i], i == 0 ? L::kBuilders : 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, 128);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = warp_uniform(*tmem_slot);
    pdl_wait();  // set-up done; the partials come from the previous kernel of the stream

    if (warp == 0) {
        // ------------------------------------------------------------------ W^UV chunks (MN-major B operand)
        const uint32_t e = elect_one();
        if (e) tma_prefetch_desc(&tmB);
        mbar_expect_tx(b_full, n_chunks * L::kBBytes, e);
        for (int c = 0; c < n_chunks; ++c)
            for (int kb = 0; kb < 2; ++kb)
                for (int nb = 0; nb < 2; ++nb)
                    tma_load_2d(b_smem + c * L::kBBytes + (kb * 2 + nb) * 8192, &tmB, nb * 64,
                                j * p.r_kv + c * L::kChunkK + kb * 64, b_full, e);
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t e = elect_one();
        constexpr uint32_t idesc = idesc_bf16(64, 128, 0, 1);
        bool ok = warp_all(mbar_wait(b_full, 0, ab, 2));
        for (int t = 0; t < n_tiles && ok; ++t) {
            if (!(ok = warp_all(mbar_wait(a_ready, t & 1, ab, 3)))) break;
            tc_fence_after();
            for (int c = 0; c < n_chunks; ++c) {
                const uint32_t a_addr = smem_u32(a_smem + c * L::kABytes);
                const uint32_t b_addr = smem_u32(b_smem + c * L::kBBytes);
#pragma unroll
                for (int kb = 0; kb < 2; ++kb)
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        umma_ss(tmem_base, desc_kmajor_sw128(a_addr + kb * 8192 + ks * 32),
                                desc_mnmajor_sw128(b_addr + kb * 16384 + ks * 2048, 8192), idesc, (c | kb | ks) != 0, e);
            }
            umma_commit(acc_full, e);
        }
    } else {
        // ------------------------------------------------------------------ builders, then epilogue
        const int q = warp & 3;         // TMEM lane quadrant of this warp (tile rows [16q, 16q + 16) in the epilogue)
        const int bw = warp - 2;        // builder warp: rows bw, bw + 16, .. of a tile
        // row gr of the group: position gr / hpb, head j * hpg + gr % hpb (head slots beyond the group's hpg heads stay empty)
        auto row_of = [&](int64_t gr, int64_t* part_row, int64_t* out_row) -> bool {
            const int64_t pos = gr / p.hpb;
            const int slot = (int)(gr % p.hpb);
            if (gr >= row0 + n_rows || slot >= p.hpg) return false;
            const int i = j * p.hpg + slot;
            const int64_t b = pos / p.s_q;
            const int pq = (int)(pos % p.s_q);
            *part_row = b * p.S * rows_per_seq + (int64_t)pq * p.h_q + i;  // split 0; + k * rows_per_seq
            *out_row = pos * p.h_q + i;
            return true;
        };
        const int chunk16 = (lane & 15) >> 1, half = lane & 1;
        uint8_t* a_lane = a_smem + (lane >> 4) * 8192;  // k-block (within a chunk) of this lane's 4 columns
        float* w_warp = sm_w + 4 * bw * L::kMaxS;       // weights of this warp's four rows
        bool ok = true;
        for (int t = 0; t < n_tiles; ++t) {
            const int64_t tile0 = row0 + (int64_t)t * L::kRows;
            const int rows_here = n_rows - t * L::kRows < L::kRows ? n_rows - t * L::kRows : L::kRows;
            // weights of this warp's rows over the S slots: eight lanes per row, lane slots k = (lane & 7) + 8 i
            int64_t pr = 0, orow = 0;
            {
                const int k0 = lane & 7;
                const bool have = row_of(tile0 + bw + 16 * (lane >> 3), &pr, &orow);
                float v[L::kMaxS / 8];
                float M = -INFINITY, den = 0.f;
#pragma unroll
                for (int i = 0; i < L::kMaxS / 8; ++i) {
                    const int k = k0 + 8 * i;
                    v[i] = have && k < p.S ? __ldg(p.lse_part + pr + (int64_t)k * rows_per_seq) : -INFINITY;
                    M = fmaxf(M, v[i]);
                }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
#pragma unroll
                for (int i = 0; i < L::kMaxS / 8; ++i) {
                    v[i] = M > -INFINITY ? expf(v[i] - M) : 0.f;
                    den += v[i];
                }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
                const float inv = den > 0.f ? 1.f / den : 0.f;
                __syncwarp();  // the previous tile's weights have been read
#pragma unroll
                for (int i = 0; i < L::kMaxS / 8; ++i)
                    if (k0 + 8 * i < p.S) w_warp[(lane >> 3) * L::kMaxS + k0 + 8 * i] = inv == 0.f ? 0.f : v[i] * inv;
                if (have && k0 == 0 && p.lse != nullptr) p.lse[orow] = den > 0.f ? M + logf(den) : -INFINITY;
            }
            __syncwarp();
#pragma unroll 1
            for (int u = 0; bw + 16 * u < rows_here; ++u) {
                const int tr = bw + 16 * u;
                const float* w_row = w_warp + u * L::kMaxS;
                const float* src = p.o_part + __shfl_sync(0xffffffffu, pr, u * 8) * p.r_kv + 4 * lane;
                // live slots of the row, one bit each (an empty slot's partial may hold anything and is not fetched)
                uint64_t live = __ballot_sync(0xffffffffu, lane < p.S && w_row[lane] != 0.f);
                if (p.S > 32) live |= (uint64_t)__ballot_sync(0xffffffffu, lane + 32 < p.S && w_row[lane + 32] != 0.f) << 32;
                float4 acc[L::kMaxChunks];
#pragma unroll
                for (int c = 0; c < L::kMaxChunks; ++c) acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
                while (live != 0) {
                    float w[3];
                    float4 x[3][L::kMaxChunks];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const int k = live != 0 ? __ffsll((long long)live) - 1 : -1;
                        live &= live - 1;  // (0 stays 0)
                        w[a] = k >= 0 ? w_row[k] : 0.f;
                        if (k >= 0) {
#pragma unroll
                            for (int c = 0; c < L::kMaxChunks; ++c)
                                if (c < n_chunks) x[a][c] = ld_partial4(src + (int64_t)k * rows_per_seq * p.r_kv + c * L::kChunkK);
                        }
                    }
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        if (w[a] != 0.f) {
#pragma unroll
                            for (int c = 0; c < L::kMaxChunks; ++c)
                                if (c < n_chunks) {
                                    acc[c].x = fmaf(w[a], x[a][c].x, acc[c].x);
                                    acc[c].y = fmaf(w[a], x[a][c].y, acc[c].y);
                                    acc[c].z = fmaf(w[a], x[a][c].z, acc[c].z);
                                    acc[c].w = fmaf(w[a], x[a][c].w, acc[c].w);
                                }
                        }
                }
#pragma unroll
                for (int c = 0; c < L::kMaxChunks; ++c)
                    if (c < n_chunks) {
                        uint2 v;
                        v.x = pack_bf16(acc[c].x, acc[c].y);
                        v.y = pack_bf16(acc[c].z, acc[c].w);
                        *reinterpret_cast<uint2*>(a_lane + c * L::kABytes + tr * 128 + ((chunk16 ^ (tr & 7)) << 4) + half * 8) = v;
                    }
            }
            fence_proxy_async_smem();  // generic-proxy writes of A -> visible to the tensor core
            tc_fence_before();         // (and this warp's reads of the previous tile's accumulator are done)
            __syncwarp();
            if (lane == 0) mbar_arrive(a_ready);
            // epilogue: TMEM lane = tile row; four warps per lane quadrant, 32 output columns each
            ok = __all_sync(0xffffffffu, mbar_wait(acc_full, t & 1, ab, 5));
            if (!ok) break;
            tc_fence_after();
            const int tr = q * 16 + (lane & 15), c0 = 32 * (bw >> 2);
            int64_t part_row = 0;
            const bool valid = lane < 16 && row_of(tile0 + tr, &part_row, &orow);  // lanes 16-31 of a quadrant hold no row
            uint32_t v[32];
            tmem_ld32(tmem_addr(tmem_base, q * 32, c0), v);
            tmem_wait_ld();
            if (valid) {
                uint4* d4 = reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.out) + orow * 128 + c0);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    uint4 o;
                    o.x = pack_bf16(__uint_as_float(v[8 * i + 0]), __uint_as_float(v[8 * i + 1]));
                    o.y = pack_bf16(__uint_as_float(v[8 * i + 2]), __uint_as_float(v[8 * i + 3]));
                    o.z = pack_bf16(__uint_as_float(v[8 * i + 4]), __uint_as_float(v[8 * i + 5]));
                    o.w = pack_bf16(__uint_as_float(v[8 * i + 6]), __uint_as_float(v[8 * i + 7]));
                    d4[i] = o;
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, 128);
}

}  // namespace tc
}  // namespace gqla
