// esp_spgemm: Y = X . P . W_s^T on the 5th-generation tensor cores with the sparse-operand MMA
// ("Efficient Sparse-GEMM Implementation": the product every pruned linear layer runs).
//
// Orientation.  The sparse operand must be the MMA's A operand, so each CTA computes a tile of Y^T:
//   D[feature (128 TMEM lanes), token (TMEM columns)] += Wc[feature, k/2] (sparse, metadata in TMEM) * Xp[k, token]
// The compressed weight arrives as pre-swizzled 18 KB tiles (16 KB values + 2 KB metadata), one bulk
// async copy per pipeline stage; the metadata is copied shared -> tensor memory with tcgen05.cp right
// before the four K=32 MMAs of a 128-channel tile.  The permutation P is applied while the X tile is
// brought into shared memory (element gather in this file), never as a separate pass over X.
// K is split across the CTAs of a thread-block cluster; partial tiles are summed in slice order through
// distributed shared memory, so no global scratch is used and the result is deterministic.
#include "esp_common.cuh"

#include <cuda.h>

#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <string>

#include <dlfcn.h>

#include "spgemm_device.cuh"

namespace esp {
namespace {

template <int BN, int STAGES>
struct GatherSmem {
    static constexpr int kWBytes = STAGES * kTileBytes;
    static constexpr int kXStage = BN * 256;                   // BN tokens x 128 channels fp16
    static constexpr int kXBytes = STAGES * kXStage;
    static constexpr int kStageArea = kWBytes + kXBytes;
    static constexpr int kReduceBytes = BN * 128 * 4;          // fp32 partial tile, aliases the stage area
    static constexpr int kMain = kStageArea > kReduceBytes ? kStageArea : kReduceBytes;
    static constexpr int kBarOff = kMain;                      // barriers, TMEM slot, abort flag
    static constexpr int kTotal = kBarOff + 256 + 1024;        // + slack for 1024-byte alignment of the base
};

// --------------------------------------------------------------------------------------------------
// Gather kernel: any M, either X layout; the X tile is gathered element-wise through the permutation by
// four warps.  Used for decode shapes (X is tiny and cache resident, the weight stream is the cost).
// grid (feature tiles, token tiles, split_k), cluster (1, 1, split_k), block 192:
//   warp 0 lane 0  weight-tile producer (bulk async copies)      warp 1 lane 0  MMA issuer
//   warps 2..5     X gather producers, then epilogue (one TMEM lane quarter each)
// --------------------------------------------------------------------------------------------------
template <int BN, int STAGES>
__global__ void __launch_bounds__(192) spgemm_gather_kernel(const GemmParams p) {
    using L = GatherSmem<BN, STAGES>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t w_base = sbase, x_base = sbase + L::kWBytes;
    const uint32_t bar_base = sbase + L::kBarOff;
    auto full_w = [&](int s) { return bar_base + 8u * s; };
    auto full_x = [&](int s) { return bar_base + 8u * (STAGES + s); };
    auto empty = [&](int s) { return bar_base + 8u * (2 * STAGES + s); };
    const uint32_t accum_bar = bar_base + 8u * (3 * STAGES);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + L::kBarOff + 8 * (3 * STAGES + 1));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + L::kBarOff + 8 * (3 * STAGES + 1) + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ft = blockIdx.x, tok0 = blockIdx.y * BN;
    const int split = (int)gridDim.z, slice = (int)blockIdx.z;
    const int kt_begin = slice * p.k_tiles_per_split;
    const int kt_end = min(p.k_tiles, kt_begin + p.k_tiles_per_split);
    const int nk = max(0, kt_end - kt_begin);
    constexpr uint32_t kTmemCols = tmem_cols_for(BN);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_w(s), 1);
            mbar_init(full_x(s), 4);
            mbar_init(empty(s), 1);
        }
        mbar_init(accum_bar, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 0) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            const uint8_t *src = p.packed + ((long)ft * p.k_tiles + kt_begin) * kTileBytes;
            for (int it = 0; it < nk; ++it) {
                const int s = it % STAGES;
                const uint32_t ph = (uint32_t)(it / STAGES) & 1u;
                if (!mbar_wait(empty(s), ph ^ 1u, abort_flag)) break;
                mbar_arrive_expect_tx(full_w(s), kTileBytes);
                bulk_load(w_base + s * kTileBytes, src + (long)it * kTileBytes, kTileBytes, full_w(s));
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = instr_desc_sparse_f16(128, BN, 0);
            for (int it = 0; it < nk; ++it) {
                const int s = it % STAGES;
                const uint32_t ph = (uint32_t)(it / STAGES) & 1u;
                if (!mbar_wait(full_w(s), ph, abort_flag)) break;
                if (!mbar_wait(full_x(s), ph, abort_flag)) break;
                tc_fence_after();
                const uint32_t wa = w_base + s * kTileBytes;
                const uint32_t xa = x_base + s * L::kXStage;
                const uint32_t e_col = BN + (it & 1) * 4;
                tc_copy_128x128b(tmem + e_col, smem_desc(wa + kTileValBytes, 0, 128, kLayoutNone));
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t col = e_col + j;
                    const uint64_t ad = smem_desc(wa + j * 32, 16, 1024, kLayoutSw128);
                    const uint64_t bd = smem_desc(xa + (j >> 1) * (BN * 128) + (j & 1) * 64, 16, 1024, kLayoutSw128);
                    tc_mma_sparse_f16(tmem, ad, bd, tmem + (col & ~1u), idesc | (col & 1u), (it > 0 || j > 0) ? 1u : 0u);
                }
                tc_commit(empty(s));
            }
            tc_commit(accum_bar);
        }
    } else {
        // ---- X gather: thread g owns channel chunk (g & 15) of tokens (g >> 4) + 8 i
        const int g = threadIdx.x - 64;
        const int chunk = g & 15;
        bool alive = true;
        for (int it = 0; it < nk && alive; ++it) {
            const int s = it % STAGES;
            const uint32_t ph = (uint32_t)(it / STAGES) & 1u;
            if (!mbar_wait(empty(s), ph ^ 1u, abort_flag)) { alive = false; break; }
            const int kc = (kt_begin + it) * kTileK + chunk * 8;
            int th[8];
            if (kc + 8 <= p.K && p.perm) {
                const int4 a = __ldg(reinterpret_cast<const int4 *>(p.perm + kc));
                const int4 b = __ldg(reinterpret_cast<const int4 *>(p.perm + kc + 4));
                th[0] = a.x; th[1] = a.y; th[2] = a.z; th[3] = a.w;
                th[4] = b.x; th[5] = b.y; th[6] = b.z; th[7] = b.w;
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) th[e] = (kc + e < p.K) ? (p.perm ? p.perm[kc + e] : kc + e) : -1;
            }
            uint8_t *xs = smem + L::kWBytes + s * L::kXStage + (chunk >> 3) * (BN * 128);
            const int q = chunk & 7;
            for (int row = g >> 4; row < BN; row += 8) {
                const int t = tok0 + row;
                uint4 v = make_uint4(0, 0, 0, 0);
                if (t < p.M) {
                    uint16_t h[8];
                    const uint16_t *xb = reinterpret_cast<const uint16_t *>(p.X);
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        long off = p.x_channel_major ? ((long)th[e] * p.ldx + t) : ((long)t * p.ldx + th[e]);
                        h[e] = th[e] >= 0 ? __ldg(xb + off) : (uint16_t)0;
                    }
                    v.x = h[0] | ((uint32_t)h[1] << 16);
                    v.y = h[2] | ((uint32_t)h[3] << 16);
                    v.z = h[4] | ((uint32_t)h[5] << 16);
                    v.w = h[6] | ((uint32_t)h[7] << 16);
                }
                *reinterpret_cast<uint4 *>(xs + row * 128 + ((q ^ (row & 7)) << 4)) = v;
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(full_x(s));
        }
        // ---- epilogue: TMEM lane quarter (warp & 3)
        const int quarter = warp & 3;
        const int f_local = quarter * 32 + lane;
        const long feature = (long)ft * 128 + f_local;
        bool ok = alive && (nk == 0 || mbar_wait(accum_bar, 0, abort_flag));
        tc_fence_after();
        float *stage_f32 = reinterpret_cast<float *>(smem);
        const float bias_f = epilogue_bias(p, feature);
#pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 16) {
            uint32_t v[16];
            if (nk > 0) {
                tmem_load_16(tmem + ((uint32_t)(quarter * 32) << 16) + c0, v);
            } else {
#pragma unroll
                for (int e = 0; e < 16; ++e) v[e] = 0;
            }
            if (split == 1) {
                if (ok && feature < p.N) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int t = tok0 + c0 + e;
                        if (t < p.M) {
                            const float y = epilogue_apply(__uint_as_float(v[e]), bias_f, p.act);
                            if (p.out_f32) reinterpret_cast<float *>(p.Y)[(long)t * p.ldy + feature] = y;
                            else reinterpret_cast<__half *>(p.Y)[(long)t * p.ldy + feature] = __float2half_rn(y);
                        }
                    }
                }
            } else {
#pragma unroll
                for (int e = 0; e < 16; ++e) stage_f32[(c0 + e) * 128 + f_local] = __uint_as_float(v[e]);
            }
        }
        tc_fence_before();
    }

    if (split > 1) {
        // all partial tiles are in shared memory: sum them in slice order, each CTA finishing 1/split of the tokens
        cluster_sync_all();
        const uint32_t rank = cluster_ctarank();
        const bool ok = (*abort_flag == 0);
        for (int idx = threadIdx.x; idx < BN * 128; idx += 192) {
            const int row = idx >> 7, f_local = idx & 127;
            if ((row % split) != (int)rank) continue;
            const int t = tok0 + row;
            const long feature = (long)ft * 128 + f_local;
            if (t >= p.M || feature >= p.N) continue;
            float acc = 0.f;
            for (int r = 0; r < split; ++r) acc += ld_dsmem_f32(sbase + (uint32_t)idx * 4u, (uint32_t)r);
            if (ok) {
                acc = epilogue_value(p, acc, feature);
                if (p.out_f32) reinterpret_cast<float *>(p.Y)[(long)t * p.ldy + feature] = acc;
                else reinterpret_cast<__half *>(p.Y)[(long)t * p.ldy + feature] = __float2half_rn(acc);
            }
        }
        cluster_sync_all();
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

template <int BN, int STAGES>
esp_status_t launch_gather(const GemmParams &p, int f_tiles, int t_tiles, int split, cudaStream_t stream) {
    using L = GatherSmem<BN, STAGES>;
    auto kern = spgemm_gather_kernel<BN, STAGES>;
    ESP_CUDA_OK(ensure_dynamic_smem((const void *)kern, L::kTotal));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(f_tiles, t_tiles, split);
    cfg.blockDim = dim3(192);
    cfg.dynamicSmemBytes = L::kTotal;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = split;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    ESP_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, p));
    return ESP_OK;
}


// --------------------------------------------------------------------------------------------------
// TMA kernel: large token counts (prefill), channel-major X.
// The X tile of a stage is 128 permuted channels x BN tokens.  Channel rows are fetched by the tensor
// memory unit four arbitrary rows at a time (tile::gather4, row indices = 4 consecutive entries of the
// permutation), 64 tokens (128 bytes) per row, landing 128-byte swizzled as an MN-major B operand: the
// permutation costs nothing beyond the loads themselves and no permuted copy of X exists anywhere.
// grid (feature tiles, token tiles, split_k), cluster (1,1,split_k), block 192:
//   warp 0  producer: lane 0 issues the weight-tile bulk copy, all lanes issue gather4 row loads
//   warp 1  lane 0 issues tcgen05.cp (metadata) + 4 sparse MMAs per stage
//   warps 2..5  epilogue
// --------------------------------------------------------------------------------------------------
__device__ __forceinline__ void tma_gather4(uint32_t dst, const CUtensorMap *map, int x, int r0, int r1, int r2, int r3,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cta.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
        "l"(map), "r"(x), "r"(r0), "r"(r1), "r"(r2), "r"(r3), "r"(bar)
        : "memory");
}

template <int BN>
struct TmaCfg {
    static constexpr int kXStage = 128 * BN * 2;
    static constexpr int kStage = kTileBytes + kXStage;
    static constexpr int kStages = (BN == 256) ? 2 : (BN == 128) ? 4 : 6;
    static constexpr int kBarOff = kStages * kStage;
    static constexpr int kTotal = kBarOff + 256 + 1024;
};

template <int BN>
__global__ void __launch_bounds__(192) spgemm_tma_kernel(const GemmParams p, const __grid_constant__ CUtensorMap xmap) {
    using L = TmaCfg<BN>;
    constexpr int STAGES = L::kStages;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar_base = sbase + L::kBarOff;
    auto full = [&](int s) { return bar_base + 8u * s; };
    auto empty = [&](int s) { return bar_base + 8u * (8 + s); };
    const uint32_t accum_bar = bar_base + 8u * 16;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + L::kBarOff + 8 * 17);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + L::kBarOff + 8 * 17 + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ft = blockIdx.x, tok0 = blockIdx.y * BN;
    const int split = (int)gridDim.z, slice = (int)blockIdx.z;
    const int kt_begin = slice * p.k_tiles_per_split;
    const int kt_end = min(p.k_tiles, kt_begin + p.k_tiles_per_split);
    const int nk = max(0, kt_end - kt_begin);
    constexpr uint32_t kTmemCols = tmem_cols_for(BN);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
        mbar_init(accum_bar, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 0) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        const uint8_t *w_src = p.packed + ((long)ft * p.k_tiles + kt_begin) * kTileBytes;
        bool alive = true;
        for (int it = 0; it < nk && alive; ++it) {
            const int s = it % STAGES;
            const uint32_t ph = (uint32_t)(it / STAGES) & 1u;
            // this lane's permutation entries: rows 4*lane .. 4*lane+3 of the stage
            const int kpos = (kt_begin + it) * kTileK + lane * 4;
            int4 rows;
            if (kpos + 4 <= p.K && p.perm) {
                rows = __ldg(reinterpret_cast<const int4 *>(p.perm + kpos));
            } else {
                int r[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) r[e] = (kpos + e < p.K) ? (p.perm ? __ldg(p.perm + kpos + e) : kpos + e) : p.K;   // K = out of range: zero fill
                rows = make_int4(r[0], r[1], r[2], r[3]);
            }
            if (!mbar_wait(empty(s), ph ^ 1u, abort_flag)) { alive = false; }
            alive = __all_sync(0xFFFFFFFFu, alive);
            if (!alive) break;
            const uint32_t stage = sbase + s * L::kStage;
            if (lane == 0) {
                mbar_arrive_expect_tx(full(s), L::kStage);
                bulk_load(stage, w_src + (long)it * kTileBytes, kTileBytes, full(s));
            }
            __syncwarp();
#pragma unroll
            for (int tb = 0; tb < BN / 64; ++tb)
                tma_gather4(stage + kTileBytes + tb * 16384 + lane * 512, &xmap, tok0 + tb * 64, rows.x, rows.y, rows.z, rows.w, full(s));
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = instr_desc_sparse_f16(128, BN, 1);
            for (int it = 0; it < nk; ++it) {
                const int s = it % STAGES;
                const uint32_t ph = (uint32_t)(it / STAGES) & 1u;
                if (!mbar_wait(full(s), ph, abort_flag)) break;
                tc_fence_after();
                const uint32_t wa = sbase + s * L::kStage;
                const uint32_t xa = wa + kTileBytes;
                const uint32_t e_col = BN + (it & 1) * 4;
                tc_copy_128x128b(tmem + e_col, smem_desc(wa + kTileValBytes, 0, 128, kLayoutNone));
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t col = e_col + j;
                    const uint64_t ad = smem_desc(wa + j * 32, 16, 1024, kLayoutSw128);
                    const uint64_t bd = smem_desc(xa + j * 4096, 16384, 1024, kLayoutSw128);
                    tc_mma_sparse_f16(tmem, ad, bd, tmem + (col & ~1u), idesc | (col & 1u), (it > 0 || j > 0) ? 1u : 0u);
                }
                tc_commit(empty(s));
            }
            tc_commit(accum_bar);
        }
    } else {
        const int quarter = warp & 3;
        const int f_local = quarter * 32 + lane;
        const long feature = (long)ft * 128 + f_local;
        const bool ok = (nk == 0 || mbar_wait(accum_bar, 0, abort_flag));
        tc_fence_after();
        float *stage_f32 = reinterpret_cast<float *>(smem);
        const float bias_f = epilogue_bias(p, feature);
#pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 16) {
            uint32_t v[16];
            if (nk > 0) {
                tmem_load_16(tmem + ((uint32_t)(quarter * 32) << 16) + c0, v);
            } else {
#pragma unroll
                for (int e = 0; e < 16; ++e) v[e] = 0;
            }
            if (split == 1) {
                if (ok && feature < p.N) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int t = tok0 + c0 + e;
                        if (t < p.M) {
                            const float y = epilogue_apply(__uint_as_float(v[e]), bias_f, p.act);
                            if (p.out_f32) reinterpret_cast<float *>(p.Y)[(long)t * p.ldy + feature] = y;
                            else reinterpret_cast<__half *>(p.Y)[(long)t * p.ldy + feature] = __float2half_rn(y);
                        }
                    }
                }
            } else {
#pragma unroll
                for (int e = 0; e < 16; ++e) stage_f32[(c0 + e) * 128 + f_local] = __uint_as_float(v[e]);
            }
        }
        tc_fence_before();
    }

    if (split > 1) {
        cluster_sync_all();
        const uint32_t rank = cluster_ctarank();
        const bool ok = (*abort_flag == 0);
        for (int idx = threadIdx.x; idx < BN * 128; idx += 192) {
            const int row = idx >> 7, f_local = idx & 127;
            if ((row % split) != (int)rank) continue;
            const int t = tok0 + row;
            const long feature = (long)ft * 128 + f_local;
            if (t >= p.M || feature >= p.N) continue;
            float acc = 0.f;
            for (int r = 0; r < split; ++r) acc += ld_dsmem_f32(sbase + (uint32_t)idx * 4u, (uint32_t)r);
            if (ok) {
                acc = epilogue_value(p, acc, feature);
                if (p.out_f32) reinterpret_cast<float *>(p.Y)[(long)t * p.ldy + feature] = acc;
                else reinterpret_cast<__half *>(p.Y)[(long)t * p.ldy + feature] = __float2half_rn(acc);
            }
        }
        cluster_sync_all();
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}


// --------------------------------------------------------------------------------------------------
// Streaming kernel: every token count, channel-major X.  A stage holds one compressed weight tile
// (18 KB, one bulk asynchronous copy) and the matching X tile: 128 permuted channel rows x BN tokens,
// fetched by four producer warps with 16-byte asynchronous copies (cp.async) that complete on the stage's
// mbarrier, landing swizzled as an MN-major B operand.  (Measured on B200: the tensor memory unit retires one
// four-row gather per ~60 clocks, 8.5 B/clk per SM, far below what the MMA consumes; plain asynchronous row
// copies are not bound by that.)
//
// Decode shapes (BN = 16 / 32 / 64) are bound by the HBM stream of weight tiles, so everything is arranged
// to get those copies in flight at once: the first weight tiles are issued by thread 0 right after it has
// initialised the barriers, before tensor memory is allocated and before the CTA's first barrier; the grid is
// sized so that all CTAs are resident together (no second wave); and with `static_weights` the kernel is
// launched as a programmatic dependent of the preceding kernel on the stream, so this prologue -- which
// touches only the weights and the permutation -- overlaps the predecessor's tail, and only the X rows
// wait for it (griddepcontrol.wait).
//
// K is split across the CTAs of a cluster.  Partial tiles are reduced by pushing: the tile's tokens are dealt to the
// cluster ranks in contiguous runs of `cnt4` rows (a multiple of 4, so that four accumulator columns always go to one
// owner as one 16-byte store); every CTA sends its fp32 partial rows straight into the owner's shared memory with
// asynchronous remote stores (slot = sender's rank) that complete on the owner's mbarrier; the owner adds the slots in
// rank order -- deterministic, no global scratch.  Token tiles up to 32 keep a receive area of their own and push as
// soon as their accumulator is complete; wider tiles, whose partials would crowd out the ring, receive into the ring
// itself once a cluster barrier has told every CTA that all MMAs of the cluster are done reading it.  (Measured on
// 4096 x 4096 at 128 tokens: owners pulling the rows from their peers with remote loads took 8.4 us for 64 KB per CTA;
// element-wise pushes for slice counts that are not a power of two took 10 us at 32 tokens.  The 16-byte pushes take
// about 1.5 us.)
//
// Token-major X without a transposing launch in front of the product (whose 3 us lie on the path from one layer's output to the next
// one's input, and which costs the host 2 us):
//   kXDirect, one or two tokens  a producer thread loads its channel's elements of each stage straight from X, kXAhead stages ahead;
//   kXCluster, small weights     the cluster's slices together span all channels: each CTA reads ITS contiguous range of channels of
//                                the tile's tokens (16-byte loads along the channels), transposes it in registers into an area in
//                                shared memory [8-token chunk][channel][16 bytes], and a stage's permuted channel rows are fetched from
//                                whichever CTA of the cluster holds the channel, 16 bytes at a time, kXAhead stages ahead.
// grid (feature tiles, token tiles, split_k), cluster (1,1,split_k), block 192:
//   warp 0 lane 0  weight-tile producer        warp 1  tensor-memory allocation; lane 0: tcgen05.cp + sparse MMAs
//   warps 2..5     X row producers, then epilogue (one quarter of the accumulator lanes each)
// --------------------------------------------------------------------------------------------------
template <int BN>
struct StreamCfg {
    static constexpr int kRowBytes = BN >= 64 ? 128 : BN * 2;        // one channel row inside a block of <= 64 tokens
    static constexpr int kTokBlocks = BN >= 64 ? BN / 64 : 1;
    static constexpr int kChunks = kRowBytes / 16;                   // 16-byte pieces per row and block
    static constexpr int kBlockBytes = 128 * kRowBytes;              // 128 channel rows of one token block
    static constexpr int kXStage = 128 * BN * 2;
    static constexpr int kStage = kTileBytes + kXStage;              // a multiple of 1024
    static constexpr uint32_t kLayout = BN >= 64 ? 2u : BN == 32 ? 4u : 6u;   // 128 / 64 / 32-byte swizzle
    static constexpr int kSwzShift = BN >= 64 ? 0 : BN == 32 ? 1 : 2;         // row bits that feed the XOR
    static constexpr bool kEarlyPush = BN <= 32;                     // partial rows pushed into a receive area of their own
    // 16-byte asynchronous row copies deliver 25 / 44 / 60 GB/s per SM from 128 / 256 / 512 threads: wide X tiles get
    // sixteen producer warps, narrow ones (little X per weight tile) four
    static constexpr int kProd = BN >= 64 ? 512 : 128;
    static constexpr int kThreads = 64 + kProd;
};
// Rows of a token tile that one cluster rank owns in the K-slice reduction (a multiple of 4; rank o owns rows
// [o * cnt4, (o + 1) * cnt4) of the tile, clipped to the tile).
__host__ __device__ inline int stream_cnt4(int bn, int split) { return (((bn + split - 1) / split) + 3) & ~3; }
// Pushed partials at one owner: [sender][group of 4 rows][128 features][4 rows] fp32.
inline size_t stream_push_bytes(int bn, int split) { return split > 1 ? (size_t)split * stream_cnt4(bn, split) * 512 : 0; }
inline size_t stream_recv_bytes(int bn, int split) { return bn <= 32 ? stream_push_bytes(bn, split) : 0; }   // beside the ring
// Token-major X: how the kernel gets it (see the comment above).
constexpr int kXChannelMajor = 0, kXDirect = 1, kXCluster = 2;
constexpr int kXDirectTokens = 2, kXAreaMax = 48 * 1024;
inline int stream_x_area_bytes(int bn, int M, int k_tiles_per_split) { return k_tiles_per_split * kTileK * 16 * (((M < bn ? M : bn) + 7) / 8); }
inline size_t stream_smem_bytes(int bn, int stages, int split, int x_area) {
    size_t ring = (size_t)stages * (kTileBytes + 256 * bn);
    if (bn > 32 && ring < stream_push_bytes(bn, split)) ring = stream_push_bytes(bn, split);   // wide tiles receive into the ring
    return ring + stream_recv_bytes(bn, split) + (size_t)x_area + kPermRing * 512 + 512 + 1024;
}

// XMODE: kernels of their own, so that the registers of the token-major producers cost the channel-major form no residency.
// (Registers: two CTAs of 576 threads share an SM, 56 each; a 256-token tile has an SM to itself; of the narrow tiles, whose shared memory lets
// two to four CTAs share one, four and three.  Bounded to 56 as well, a narrow tile's X loop lost up to 10 %: 4096 x 4096 at 16 tokens,
// device-bound, 6.9 -> 6.45 us, 2208 x 6528 at 37 tokens 10.4 -> 9.7.  OVERLAP: launched as a dependent of the kernel before, whose tail then hides the start-up.
// The 32-token tile launched in plain stream order is left unbounded, 56 registers by the compiler's own choice: with 80 its start-up showed, 680 x 9668
// at 32 tokens 8.6 -> 9.6 us, 744 x 4408 at 60 8.6 -> 9.5; in dependent launches 80 are 1 % ahead, and for 16 tokens the two are even.)
template <int BN, int XMODE, bool OVERLAP>
__global__ void __launch_bounds__(StreamCfg<BN>::kThreads, BN == 256 ? 1 : BN >= 64 ? 2 : XMODE != kXChannelMajor ? 3 : OVERLAP ? 4 : 0) spgemm_stream_kernel(const GemmGroup grp, const int stages) {
    constexpr bool TM = XMODE != kXChannelMajor, xcluster = XMODE == kXCluster;
    using L = StreamCfg<BN>;
    // this CTA's problem: selected with constant indices so that the parameters stay in registers
    GemmParams p = grp.p[0];
    int ft_first = 0;
#pragma unroll
    for (int i = 1; i < ESP_MAX_GROUP; ++i)
        if (i < grp.count && (int)blockIdx.x >= grp.ft_start[i]) { p = grp.p[i]; ft_first = grp.ft_start[i]; }
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const int split = (int)gridDim.z, slice = (int)blockIdx.z;
    // layout (matches stream_smem_bytes): ring of stages | pushed partials (narrow tiles) | permutation ring | barriers;
    // wide tiles receive the pushed partials at the start of the ring
    const int cnt4 = stream_cnt4(BN, split);
    const uint32_t push_bytes = split > 1 ? (uint32_t)(split * cnt4 * 512) : 0u;
    uint32_t ring_bytes = (uint32_t)stages * L::kStage;
    if (!L::kEarlyPush && ring_bytes < push_bytes) ring_bytes = push_bytes;
    const uint32_t recv_off = L::kEarlyPush ? ring_bytes : 0u;
    const uint32_t xarea_off = ring_bytes + (L::kEarlyPush ? push_bytes : 0u);
    const uint32_t perm_off = xarea_off + (xcluster ? (uint32_t)p.x_area : 0u);
    const uint32_t bar_off = perm_off + kPermRing * 512;
    const uint32_t bar_base = sbase + bar_off;
    auto full = [&](int s) { return bar_base + 8u * s; };
    auto empty = [&](int s) { return bar_base + 8u * (kMaxStages + s); };
    const uint32_t accum_bar = bar_base + 8u * (2 * kMaxStages);
    const uint32_t recv_bar = bar_base + 8u * (2 * kMaxStages + 1);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + bar_off + 8 * (2 * kMaxStages + 2));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + bar_off + 8 * (2 * kMaxStages + 2) + 4);
    int *perm_s = reinterpret_cast<int *>(smem + perm_off);          // [kPermRing][128]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ft = (int)blockIdx.x - ft_first, tok0 = blockIdx.y * BN;
    const int kt_begin = slice * p.k_tiles_per_split;
    const int kt_end = min(p.k_tiles, kt_begin + p.k_tiles_per_split);
    const int nk = max(0, kt_end - kt_begin);
    constexpr uint32_t kTmemCols = tmem_cols_for(BN);
    const uint8_t *w_src = p.packed + ((long)ft * p.k_tiles + kt_begin) * kTileBytes;
    const int prefetch = min(stages, nk);
    // Image form (a workspace): a tiling pass has written the permuted, swizzled X operand of every (64-token
    // block -- BN < 64: token tile --, channel step) into the workspace; a stage's X is then one bulk copy per token
    // block instead of 16-byte row copies from every producer thread (which are limited to one 32-byte sector per clock
    // per SM).
    const bool imaged = !TM && p.ximg != nullptr;
    const int slice_ch = p.k_tiles_per_split * kTileK;                // channels per slice: channel c is held by rank c / slice_ch
    const uint32_t rank = (split > 1) ? cluster_ctarank() : 0u;
    const int owned = max(0, min(cnt4, BN - (int)rank * cnt4));      // rows of this tile that this CTA finishes

    if (threadIdx.x == 0) {
        // gather form: every X producer thread + the weight-tile copy; image form: the weight-tile copy + the X image copies
        for (int s = 0; s < stages; ++s) { mbar_init(full(s), imaged ? 2u : (uint32_t)L::kProd + 1u); mbar_init(empty(s), 1); }
        mbar_init(accum_bar, 1);
        mbar_init(recv_bar, 1);
        *abort_flag = 0;
        fence_barrier_init();
        // every sender delivers 128 features x (rows of this tile that this CTA owns) floats
        if (split > 1) mbar_arrive_expect_tx(recv_bar, (uint32_t)(split * owned * 512));
    }
    if (warp == 0) {
        // The weight stream starts now: nothing below is needed for these copies.  Lane s owns stage s (bulk copies
        // issued by one thread complete one after the other, copies of different threads overlap).
        __syncwarp();
        if (lane < prefetch) {
            mbar_arrive_expect_tx(full(lane), kTileBytes);
            bulk_load(sbase + lane * L::kStage, w_src + (long)lane * kTileBytes, kTileBytes, full(lane));
        }
    }
    if (warp == 1) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    if (warp >= 2 && warp < 6 && !imaged) {
        // permutation entries of the first stages, all loads in flight together (the X addresses depend on them)
        const int g = threadIdx.x - 64;
        int pre[kPermRing];
#pragma unroll
        for (int it = 0; it < kPermRing; ++it) {
            const int kpos = (kt_begin + it) * kTileK + g;
            pre[it] = (it < nk && kpos < p.K) ? (p.perm ? __ldg(p.perm + kpos) : kpos) : -1;
        }
#pragma unroll
        for (int it = 0; it < kPermRing; ++it) perm_s[it * 128 + g] = pre[it];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (split > 1 && !(xcluster && warp >= 2)) cluster_arrive();       // every CTA of the cluster is running and has its barriers set up
    grid_launch_dependents();

    // Cluster barrier protocol (split > 1): phase A = "every CTA has its barriers set up" (arrived above; with token-major X also "its
    // channels are in the X area", arrived by the producers, where the cluster shares X); wide tiles add phase B = "every CTA's MMAs are done with the ring",
    // shared X phase Z = "this CTA reads no other's X area any more" (waited for before the exit).  Every thread takes part in
    // every phase, whatever happened to it.
    if (warp == 0) {
        // (later weight tiles are issued by the X producer warps below, right after they have seen the stage's `empty`)
        if (split > 1) {
            cluster_wait();
            if (!L::kEarlyPush) { cluster_arrive(); cluster_wait(); }
            if (xcluster) cluster_arrive();
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = instr_desc_sparse_f16(128, BN, 1);
            for (int it = 0; it < nk; ++it) {
                const int s = it % stages;
                const uint32_t ph = (uint32_t)(it / stages) & 1u;
                if (!mbar_wait(full(s), ph, abort_flag)) break;
                fence_async_smem();          // rows written by cp.async (generic proxy) -> read by the MMA (async proxy)
                tc_fence_after();
                const uint32_t wa = sbase + s * L::kStage;
                const uint32_t xa = wa + kTileBytes;
                const uint32_t e_col = BN + (it & 1) * 4;
                tc_copy_128x128b(tmem + e_col, smem_desc(wa + kTileValBytes, 0, 128, kLayoutNone));
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t col = e_col + j;
                    const uint64_t ad = smem_desc(wa + j * 32, 16, 1024, kLayoutSw128);
                    const uint64_t bd = (BN >= 64) ? smem_desc(xa + j * 4096, L::kBlockBytes, 1024, kLayoutSw128)
                                                   : smem_desc(xa + j * 32 * L::kRowBytes, 8 * L::kRowBytes, 8 * L::kRowBytes, L::kLayout);
                    tc_mma_sparse_f16(tmem, ad, bd, tmem + (col & ~1u), idesc | (col & 1u), (it > 0 || j > 0) ? 1u : 0u);
                }
                tc_commit(empty(s));
            }
            tc_commit(accum_bar);
        }
        __syncwarp();
        if (split > 1) {
            cluster_wait();
            if (!L::kEarlyPush) { cluster_arrive(); cluster_wait(); }
            if (xcluster) cluster_arrive();
        }
    } else {
        // ---- X producers: thread g copies the 16-byte pieces e = g, g + 128, ... of the stage's 128 rows
        const int g = threadIdx.x - 64;
        constexpr int kPieces = 128 * L::kChunks;                     // per token block
        constexpr int kPerThread = (kPieces + L::kProd - 1) / L::kProd;
        const uint16_t *xb = reinterpret_cast<const uint16_t *>(p.X);
        const bool ring_refill = nk > kPermRing;                      // long K-slices: keep the ring kPermRing stages ahead
        bool alive = true;
        int refill = -1;
        if (imaged) {
            // ---- image form: lane 0 of producer warp q feeds the ring slots s = q, q + 4, ...: the weight tile (beyond the
            // start-up ones) and the X images of the tile's 64-token blocks, each a bulk copy.  A slot always has the same
            // feeder, which therefore waits for the slot's `empty` phases one after the other (a thread that ran two phases
            // ahead of a barrier would see the older phase of the same parity as complete).  The images are written by
            // the tiling pass this kernel is a programmatic dependent of; a raised flag also says that everything before
            // that pass is complete (its CTAs waited for it), so Y may be written once any flag has been seen.
            const int q = warp - 2;
            const int h0 = (int)blockIdx.y * L::kTokBlocks;                              // first 64-token block of this tile
            const int n_blocks = BN < 64 ? 1 : min(L::kTokBlocks, 2 * ((p.M + 127) / 128) - h0);   // (64-token blocks: the pass writes whole 128-token pairs)
            if (q < 4 && lane == 0) {
                for (int it = 0; it < nk; ++it) {
                    const int s = it % stages;
                    if ((s & 3) != q) continue;
                    const uint32_t ph = (uint32_t)(it / stages) & 1u;
                    const int kt = kt_begin + it;
                    bool seen = true;
                    for (int tb = 0; tb < n_blocks; ++tb) seen = seen && xflag_wait(p.xflags + (size_t)(h0 + tb) * p.k_tiles + kt, abort_flag);
                    if (!seen) { alive = false; break; }
                    asm volatile("fence.proxy.async;" ::: "memory");   // the pass's generic-proxy writes, just acquired -> this thread's bulk read
                    if (!mbar_wait(empty(s), ph ^ 1u, abort_flag)) { alive = false; break; }
                    if (it >= prefetch) {
                        mbar_arrive_expect_tx(full(s), kTileBytes);
                        bulk_load(sbase + s * L::kStage, w_src + (long)it * kTileBytes, kTileBytes, full(s));
                    }
                    mbar_arrive_expect_tx(full(s), (uint32_t)(n_blocks * L::kBlockBytes));
                    for (int tb = 0; tb < n_blocks; ++tb)
                        bulk_load(sbase + s * L::kStage + kTileBytes + tb * L::kBlockBytes,
                                  p.ximg + ((size_t)(h0 + tb) * p.k_tiles + kt) * L::kBlockBytes, L::kBlockBytes, full(s));
                }
            }
            if (nk == 0) grid_dependency_wait();                      // (no flag to see: wait for the stream order itself)
        } else if constexpr (TM) {
            // ---- token-major X: this slice's channels into the X area, then a stage's rows from the cluster's areas
            const int chunks = (min(p.M, BN) + 7) >> 3;               // 8-token chunks of the tile that exist
            const int own_ch = nk * kTileK, area_ch = slice_ch;
            uint8_t *area = smem + xarea_off;
            // chunks beyond them: zero in every ring slot, once
            if (chunks < L::kChunks) {
                for (int i = g; i < stages * 128 * (L::kChunks - chunks); i += L::kProd) {
                    const int s = i / (128 * (L::kChunks - chunks)), q = i - s * (128 * (L::kChunks - chunks));
                    const int r = q & 127, cc = chunks + (q >> 7);
                    const int cs = cc ^ ((r >> L::kSwzShift) & (L::kChunks - 1));
                    *reinterpret_cast<uint4 *>(smem + s * L::kStage + kTileBytes + r * L::kRowBytes + (cs << 4)) = make_uint4(0u, 0u, 0u, 0u);
                }
            }
            grid_dependency_wait();                                   // X may come from the preceding kernel
            if constexpr (xcluster) {
            for (int i = g; i < (own_ch >> 3) * chunks; i += L::kProd) {
                const int blk = i % (own_ch >> 3), cc = i / (own_ch >> 3);
                const int c = kt_begin * kTileK + blk * 8, t0 = tok0 + cc * 8;
                uint4 v[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    v[t] = make_uint4(0u, 0u, 0u, 0u);
                    if (c < p.K && t0 + t < p.M) v[t] = __ldg(reinterpret_cast<const uint4 *>(xb + (long)(t0 + t) * p.ldx + c));
                }
                // 8 x 8 transposition; channel 8 b + e goes to place 8 b + (e ^ (b & 7)), so that neighbouring threads meet different banks
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const uint32_t sel = (e & 1) ? 0x7632u : 0x5410u;
                    uint32_t w[8], o[4];
#pragma unroll
                    for (int t = 0; t < 8; ++t) w[t] = (e >> 1) == 0 ? v[t].x : (e >> 1) == 1 ? v[t].y : (e >> 1) == 2 ? v[t].z : v[t].w;
#pragma unroll
                    for (int j = 0; j < 4; ++j) o[j] = __byte_perm(w[2 * j], w[2 * j + 1], sel);
                    *reinterpret_cast<uint4 *>(area + ((size_t)cc * area_ch + blk * 8 + (e ^ (blk & 7))) * 16) = make_uint4(o[0], o[1], o[2], o[3]);
                }
            }
            __syncwarp();
            if (split > 1) { cluster_arrive(); cluster_wait(); }      // phase A
            else asm volatile("bar.sync 1, %0;" ::"n"(L::kProd) : "memory");
            }
            const uint32_t area_s = sbase + xarea_off;
            const bool ring_over = nk > kPermRing;                    // (g < 128 = every producer of these tiles)
            static_assert(L::kProd == 128, "one channel row per producer");
            constexpr int kXAhead = XMODE == kXDirect ? 8 : BN == 16 ? 2 : 1;
            static_assert(kPermRing >= 2 * kXAhead, "ring of permutation entries");
            constexpr int kRegs = XMODE == kXDirect ? 1 : L::kChunks;
            uint4 ahead[kXAhead][kRegs];                              // (direct: word t = the element of token t)
            auto fetch = [&](int it, uint4 (&v)[kRegs]) {
#pragma unroll
                for (int cc = 0; cc < kRegs; ++cc) v[cc] = make_uint4(0u, 0u, 0u, 0u);
                // (a thread reads and writes its own entries of the permutation ring only)
                const int ch = it < nk ? perm_s[(it % kPermRing) * 128 + g] : -1;
                if (ch < 0) return;
                if constexpr (XMODE == kXDirect) {
                    const uint16_t *x = xb + ch;
                    v[0].x = __ldg(x);
                    if (p.M > 1) v[0].y = __ldg(x + p.ldx);
                } else {
                    const int owner = ch / slice_ch, local = ch - owner * slice_ch;
                    const uint32_t at = area_s + (uint32_t)((local ^ ((local >> 3) & 7)) * 16);
                    const uint32_t remote = split > 1 ? map_to_rank(at, (uint32_t)owner) : at;
#pragma unroll
                    for (int cc = 0; cc < L::kChunks; ++cc)
                        if (cc < chunks)
                            asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
                                         : "=r"(v[cc].x), "=r"(v[cc].y), "=r"(v[cc].z), "=r"(v[cc].w)
                                         : "r"(remote + (uint32_t)(cc * area_ch * 16))
                                         : "memory");
                }
            };
#pragma unroll
            for (int u = 0; u < kXAhead; ++u) fetch(u, ahead[u]);
            for (int it0 = 0; it0 < nk; it0 += kXAhead) {
#pragma unroll
                for (int u = 0; u < kXAhead; ++u) {
                    const int it = it0 + u;
                    if (it >= nk) break;
                    const int s = it % stages;
                    const uint32_t ph = (uint32_t)(it / stages) & 1u;
                    if (alive && !mbar_wait(empty(s), ph ^ 1u, abort_flag)) alive = false;
                    if (alive) {
                        uint8_t *xs = smem + s * L::kStage + kTileBytes + g * L::kRowBytes;
                        if constexpr (XMODE == kXDirect) {
                            const uint4 e = ahead[u][0];
                            *reinterpret_cast<uint4 *>(xs + (((g >> L::kSwzShift) & (L::kChunks - 1)) << 4)) = make_uint4(e.x | (e.y << 16), 0u, 0u, 0u);
                        } else {
#pragma unroll
                            for (int cc = 0; cc < L::kChunks; ++cc)
                                if (cc < chunks) *reinterpret_cast<uint4 *>(xs + ((cc ^ ((g >> L::kSwzShift) & (L::kChunks - 1))) << 4)) = ahead[u][cc];
                        }
                        fence_async_smem();                           // generic-proxy writes -> read by the MMA
                        mbar_arrive(full(s));
                        if (it >= prefetch && lane == 0 && (warp - 2) == (s & 3)) {      // weight tile beyond the start-up ones, as below
                            mbar_arrive_expect_tx(full(s), kTileBytes);
                            bulk_load(sbase + s * L::kStage, w_src + (long)it * kTileBytes, kTileBytes, full(s));
                        }
                    }
                    if (ring_over) {                                  // the entry of stage it is used up: that of kPermRing stages on
                        if (it > 0) perm_s[((it - 1) % kPermRing) * 128 + g] = refill;
                        const int kpos = (kt_begin + it + kPermRing) * kTileK + g;
                        refill = (it + kPermRing < nk && kpos < p.K) ? (p.perm ? __ldg(p.perm + kpos) : kpos) : -1;
                    }
                    fetch(it + kXAhead, ahead[u]);
                }
            }
            __syncwarp();
            if (xcluster && split > 1) cluster_arrive();              // phase Z (waited for at the end)
        } else {
        grid_dependency_wait();                                       // X may come from the preceding kernel
        for (int it = 0; it < nk; ++it) {
            const int s = it % stages;
            const uint32_t ph = (uint32_t)(it / stages) & 1u;
            const int *pr = perm_s + (it % kPermRing) * 128;
            if (ring_refill && it > 0 && g < 128) perm_s[((it - 1) % kPermRing) * 128 + g] = refill;   // entries of stage it-1+kPermRing
            int ch[kPerThread];
#pragma unroll
            for (int i = 0; i < kPerThread; ++i) {
                const int e = g + L::kProd * i;
                ch[i] = (e < kPieces) ? pr[e / L::kChunks] : -1;
            }
            if (ring_refill) {
                asm volatile("bar.sync 1, %0;" ::"n"(L::kProd) : "memory");   // everyone has read this stage's entries
                const int kpos = (kt_begin + it + kPermRing) * kTileK + g;
                refill = (g < 128 && it + kPermRing < nk && kpos < p.K) ? (p.perm ? __ldg(p.perm + kpos) : kpos) : -1;
            }
            // (a thread whose wait gave up keeps looping without copying: the named barrier above needs every producer)
            if (alive && !mbar_wait(empty(s), ph ^ 1u, abort_flag)) alive = false;
            if (!alive) continue;
            const uint32_t xs = sbase + s * L::kStage + kTileBytes;
#pragma unroll
            for (int tb = 0; tb < L::kTokBlocks; ++tb) {
#pragma unroll
                for (int i = 0; i < kPerThread; ++i) {
                    const int e = g + L::kProd * i;
                    if (e < kPieces) {
                        const int r = e / L::kChunks, cc = e % L::kChunks;
                        const int t = tok0 + tb * 64 + cc * 8;
                        const int valid = min(8, max(0, p.M - t));
                        const bool in = ch[i] >= 0 && valid > 0;
                        const uint16_t *src = in ? xb + (long)ch[i] * p.ldx + t : xb;
                        const int cs = cc ^ ((r >> L::kSwzShift) & (L::kChunks - 1));
                        cp_async_16(xs + tb * L::kBlockBytes + r * L::kRowBytes + (cs << 4), src, in ? valid * 2 : 0);
                    }
                }
            }
            cp_async_arrive_noinc(full(s));
            // Weight tile of this stage (beyond the first `stages`, which were issued at start-up): lane 0 of producer warp
            // s % 4.  Copies issued by one thread do not overlap and lanes spinning in one warp hold each other up, so
            // the issuing duty rotates over the four producer warps, which have just seen `empty` anyway.
            if (it >= prefetch && lane == 0 && (warp - 2) == (s & 3)) {   // (one of the first four producer warps)
                mbar_arrive_expect_tx(full(s), kTileBytes);
                bulk_load(sbase + s * L::kStage, w_src + (long)it * kTileBytes, kTileBytes, full(s));
            }
        }
        }
        // ---- epilogue: warp w reads lane quarter w % 4 and the 16-column pieces (w - 2) / 4, + kProd / 128, ...  One K-slice: the
        // warps stage the tile in shared memory and store it.  Several: they push partial rows to their owners, then finish the
        // rows this CTA owns.  (All producer warps, not four, in the one-slice form: 3456 x 744 at 334 tokens 17.4 -> 10.2 us with 128-token
        // tiles, 18.2 -> 13.4 with 256.)
        const int quarter = warp & 3;
        const int f_local = quarter * 32 + lane;
        if (imaged) {
            // Almost every producer thread has been idle since the start: one of them polls the accumulator barrier, the
            // others sleep on a named barrier (hundreds of lanes polling through the main loop slow the CTA's other
            // barrier operations down).
            if (warp == (L::kProd > 128 ? 6 : 5) && lane == 31 && nk > 0) (void)mbar_wait(accum_bar, 0, abort_flag);
            __syncwarp();
            asm volatile("bar.sync 1, %0;" ::"n"(L::kProd) : "memory");
        }
        if (split == 1) {
            const bool ok = __all_sync(0xFFFFFFFFu, alive && (nk == 0 || mbar_wait(accum_bar, 0, abort_flag)));   // warp-uniform
            tc_fence_after();
            // accumulators -> shared memory [token][128 features] in the output type -> 16-byte stores
            const int esize = p.out_f32 ? 4 : 2;
            const float bias_f = epilogue_bias(p, (long)ft * 128 + f_local);
#pragma unroll 1
            for (int c0 = ((warp - 2) >> 2) * 16; c0 < BN; c0 += L::kProd / 8) {
                uint32_t v[16];
                if (nk > 0 && ok) {
                    tmem_load_16(tmem + ((uint32_t)(quarter * 32) << 16) + c0, v);
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] = 0;
                }
                if (p.out_f32) {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        reinterpret_cast<float *>(smem)[(c0 + e) * 128 + f_local] = epilogue_apply(__uint_as_float(v[e]), bias_f, p.act);
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        reinterpret_cast<__half *>(smem)[(c0 + e) * 128 + f_local] =
                            __float2half_rn(epilogue_apply(__uint_as_float(v[e]), bias_f, p.act));
                }
            }
            tc_fence_before();
            asm volatile("bar.sync 1, %0;" ::"n"(L::kProd) : "memory");
            const int row_bytes = 128 * esize;
            const int chunks_per_row = row_bytes / 16;
            const int f_valid = min(128, p.N - ft * 128);
            const bool vec_ok = (((long)p.ldy * esize) % 16 == 0) && ((reinterpret_cast<uintptr_t>(p.Y) & 15) == 0) && f_valid % (16 / esize) == 0;
            const long y0 = (long)tok0 * p.ldy + (long)ft * 128;
            const int rows = ok ? min(BN, p.M - tok0) : 0;
            if (vec_ok) {
                uint8_t *yb = reinterpret_cast<uint8_t *>(p.Y) + y0 * esize;
                for (int idx = g; idx < rows * chunks_per_row; idx += L::kProd) {
                    const int row = idx / chunks_per_row, c = idx % chunks_per_row;
                    if (c * (16 / esize) < f_valid)
                        *reinterpret_cast<uint4 *>(yb + (long)row * p.ldy * esize + c * 16) = *reinterpret_cast<const uint4 *>(smem + (size_t)row * row_bytes + c * 16);
                }
            } else if (p.out_f32) {
                store_unaligned_rows(reinterpret_cast<float *>(p.Y) + y0, p.ldy, reinterpret_cast<const float *>(smem), f_valid, rows, g >> 5, L::kProd / 32, lane);
            } else {
                store_unaligned_rows(reinterpret_cast<__half *>(p.Y) + y0, p.ldy, reinterpret_cast<const __half *>(smem), f_valid, rows, g >> 5, L::kProd / 32, lane);
            }
        } else {
            constexpr int kPushGroups = L::kProd / 128;                  // 16-column pieces pushed side by side
            const int cgrp = (warp - 2) >> 2;
            const bool ok = __all_sync(0xFFFFFFFFu, alive && (nk == 0 || mbar_wait(accum_bar, 0, abort_flag)));   // warp-uniform
            tc_fence_after();
            if (!xcluster) cluster_wait();                           // phase A: every CTA of the cluster has its barriers
            if (!L::kEarlyPush) { cluster_arrive(); cluster_wait(); }   // phase B: every CTA's MMAs are done with the ring
            const int groups = cnt4 >> 2;                            // 4-row groups per owner
#pragma unroll 1
            for (int c0 = cgrp * 16; c0 < BN; c0 += 16 * kPushGroups) {
                uint32_t v[16];
                if (nk > 0 && ok) {
                    tmem_load_16(tmem + ((uint32_t)(quarter * 32) << 16) + c0, v);
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] = 0;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int row = c0 + 4 * j;
                    const int owner = row / cnt4, rg = (row - owner * cnt4) >> 2;
                    const uint32_t local = sbase + recv_off + (uint32_t)((((int)rank * groups + rg) * 128 + f_local) * 16);
                    st_async_v4(map_to_rank(local, (uint32_t)owner), v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3],
                                map_to_rank(recv_bar, (uint32_t)owner));
                }
            }
            tc_fence_before();
            const bool got = mbar_wait_cluster(recv_bar, 0, abort_flag);
            const bool fine = got && (*abort_flag == 0);
            const float4 *recv = reinterpret_cast<const float4 *>(smem + recv_off);
            const int f_valid = min(128, p.N - ft * 128);
            for (int q = g; q < (owned >> 2) * 128; q += L::kProd) {
                const int rg = q >> 7, f = q & 127;
                float a[4] = {0.f, 0.f, 0.f, 0.f};
                for (int r = 0; r < split; ++r) {                    // slice order: deterministic
                    const float4 part = recv[(r * groups + rg) * 128 + f];
                    a[0] += part.x; a[1] += part.y; a[2] += part.z; a[3] += part.w;
                }
                if (!fine || f >= f_valid) continue;
                const float bias_f = epilogue_bias(p, (long)ft * 128 + f);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int t = tok0 + (int)rank * cnt4 + rg * 4 + e;
                    if (t >= p.M) continue;
                    const long o = (long)t * p.ldy + (long)ft * 128 + f;
                    const float y = epilogue_apply(a[e], bias_f, p.act);
                    if (p.out_f32) reinterpret_cast<float *>(p.Y)[o] = y;
                    else reinterpret_cast<__half *>(p.Y)[o] = __float2half_rn(y);
                }
            }
        }
    }
    if (xcluster && split > 1) cluster_wait();                        // phase Z
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// X [K, ldx] channel-major -> the streaming kernel's X stages for 16- and 32-token tiles: image (t, kt) holds channels
// perm[kt*128 .. +127] of tokens BN t .. BN t + BN - 1 as [128 rows][2 BN bytes] with the 16-byte chunk c of row r stored
// at the chunk the kernel's B descriptor expects (64-byte swizzle for 32 tokens: c ^ ((r >> 1) & 3); 32-byte swizzle for 16:
// c ^ ((r >> 2) & 1)).  Rows beyond K and tokens beyond M are zero.  grid (token tiles, k_tiles), block 256: thread -> row
// and chunk(s).  Flags as in xtile_kernel: lowered before the dependent launch may start, raised when the image is complete.
template <int BN>
__global__ void __launch_bounds__(256) xtile_narrow_kernel(const uint16_t *__restrict__ X, long ldx, int M, int K,
                                                           const int32_t *__restrict__ perm, uint8_t *__restrict__ img,
                                                           uint32_t *__restrict__ flags, int k_tiles) {
    using L = StreamCfg<BN>;
    static_assert(BN == 16 || BN == 32, "narrow tiles");
    constexpr int kPer = L::kChunks / 2;                                  // chunks per thread: 2 threads per row
    const int t = blockIdx.x, kt = blockIdx.y;
    uint8_t *dst = img + ((size_t)t * k_tiles + kt) * L::kBlockBytes;
    uint32_t *flag = flags + (size_t)t * k_tiles + kt;
    const int r = threadIdx.x >> 1, c0 = (threadIdx.x & 1) * kPer;
    const int kpos = kt * kTileK + r;
    const int ch = kpos < K ? (perm ? __ldg(perm + kpos) : kpos) : -1;
    grid_dependency_wait();                  // X may be the preceding kernel's output; the images may still be read by it
    if (threadIdx.x == 0) {
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(flag), "r"(0u) : "memory");
        __threadfence();
    }
    __syncthreads();
    grid_launch_dependents();
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int cc = c0 + i, tok = t * BN + cc * 8;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (ch >= 0 && tok < M) {
            const uint16_t *src = X + (long)ch * ldx + tok;
            if (tok + 8 <= M) {
                v = __ldg(reinterpret_cast<const uint4 *>(src));
            } else {
                uint16_t e[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) e[j] = (tok + j < M) ? __ldg(src + j) : (uint16_t)0;
                v = make_uint4(e[0] | ((uint32_t)e[1] << 16), e[2] | ((uint32_t)e[3] << 16), e[4] | ((uint32_t)e[5] << 16),
                               e[6] | ((uint32_t)e[7] << 16));
            }
        }
        const int cs = cc ^ ((r >> L::kSwzShift) & (L::kChunks - 1));
        *reinterpret_cast<uint4 *>(dst + r * L::kRowBytes + (cs << 4)) = v;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(flag), "r"(1u) : "memory");
}
inline size_t xtile_narrow_image_bytes(int M, int K, int bn) { return (size_t)((M + bn - 1) / bn) * ((K + kTileK - 1) / kTileK) * 256 * bn; }
inline size_t xtile_narrow_bytes(int M, int K, int bn) {    // images | one flag word per image
    return xtile_narrow_image_bytes(M, K, bn) + align_up((size_t)((M + bn - 1) / bn) * ((K + kTileK - 1) / kTileK) * 4, 256);
}
template <int BN>
esp_status_t launch_xtile_narrow(const GemmParams &p, uint8_t *img, uint32_t *flags, bool dependent, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((p.M + BN - 1) / BN, p.k_tiles, 1);
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    ESP_CUDA_OK(cudaLaunchKernelEx(&cfg, xtile_narrow_kernel<BN>, reinterpret_cast<const uint16_t *>(p.X), p.ldx, p.M, p.K, p.perm, img,
                                   flags, p.k_tiles));
    return ESP_OK;
}

// The kernel for these parameters.
template <int BN>
auto stream_kernel_for(int x_mode, bool dependent) {
    if constexpr (BN == 16)
        if (x_mode == kXDirect) return spgemm_stream_kernel<BN, kXDirect, true>;
    if constexpr (BN <= 32)
        if (x_mode == kXCluster) return spgemm_stream_kernel<BN, kXCluster, true>;
    if constexpr (BN == 32)
        if (!dependent) return spgemm_stream_kernel<BN, kXChannelMajor, false>;
    return spgemm_stream_kernel<BN, kXChannelMajor, true>;
}

template <int BN>
esp_status_t launch_stream(const GemmParams &p, int f_tiles, int t_tiles, int split, int stages, bool dependent,
                           cudaStream_t stream) {
    auto kern = stream_kernel_for<BN>(p.x_mode, dependent);
    const size_t smem = stream_smem_bytes(BN, stages, split, p.x_area);
    ESP_CUDA_OK(ensure_dynamic_smem((const void *)kern, (int)smem));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(f_tiles, t_tiles, split);
    cfg.blockDim = dim3(StreamCfg<BN>::kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = split;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 2 : 1;
    GemmGroup grp;
    grp.count = 1;
    for (int i = 0; i <= ESP_MAX_GROUP; ++i) grp.ft_start[i] = i == 0 ? 0 : f_tiles;
    for (int i = 0; i < ESP_MAX_GROUP; ++i) grp.p[i] = p;
    ESP_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, grp, stages));
    return ESP_OK;
}

// The same launch for a group of problems (feature tiles concatenated along grid.x).
template <int BN>
esp_status_t launch_stream_group(const GemmGroup &grp, int t_tiles, int split, int stages, bool dependent, cudaStream_t stream) {
    auto kern = stream_kernel_for<BN>(grp.p[0].x_mode, dependent);
    const size_t smem = stream_smem_bytes(BN, stages, split, grp.p[0].x_area);
    ESP_CUDA_OK(ensure_dynamic_smem((const void *)kern, (int)smem));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grp.ft_start[grp.count], t_tiles, split);
    cfg.blockDim = dim3(StreamCfg<BN>::kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = split;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 2 : 1;
    ESP_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, grp, stages));
    return ESP_OK;
}

// Clusters of `split` CTAs that the device's GPCs hold with one streaming CTA per SM, asked once per device and size.  (The occupancy
// calculator answers with one CTA per SM for these kernels whatever their size, since it cannot know how much tensor memory a CTA
// will allocate; so the packing is asked for a CTA that fills an SM, and stream_capacity_ctas counts the CTAs that share one.)
static int stream_clusters_one_per_sm(int device, int split) {
    static std::mutex mu;
    static std::map<int, int> cache;
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(device * 16 + split);
    if (it != cache.end()) return it->second;
    auto kern = stream_kernel_for<128>(kXChannelMajor, true);
    const size_t smem = stream_smem_bytes(128, 4, split, 0);
    int n = 0;
    if (ensure_dynamic_smem((const void *)kern, (int)smem) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, 1, split);
        cfg.blockDim = dim3(StreamCfg<128>::kThreads);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = split;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
    }
    if (log_plans()) fprintf(stderr, "esparse streaming clusters of %d CTAs, one CTA per SM: %d fit\n", split, n);
    return cache[device * 16 + split] = n;
}

#include "spgemm_pair.cuh"
#include "spgemm_persist.cuh"

// Tensor map over channel-major X: dim 0 = tokens (contiguous), dim 1 = channels (ldx apart); box = 64 tokens
// x 1 row (the row-gather form loads four such rows per instruction), 128-byte swizzle, zero fill outside.
inline esp_status_t make_x_tensor_map(const __half *X, int M, int K, long ldx, CUtensorMap *map) {
    EncodeTiledFn encode = nullptr;
    esp_status_t est = tensor_map_encoder(&encode);
    if (est != ESP_OK) return est;
    cuuint64_t dims[2] = {(cuuint64_t)M, (cuuint64_t)K};
    cuuint64_t strides[1] = {(cuuint64_t)ldx * 2};
    cuuint32_t box[2] = {64, 1};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half *>(X), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? ESP_OK : ESP_ERR_CUDA;
}

template <int BN>
esp_status_t launch_tma(const GemmParams &p, int f_tiles, int t_tiles, int split, cudaStream_t stream) {
    using L = TmaCfg<BN>;
    CUtensorMap map;
    esp_status_t st = make_x_tensor_map(p.X, p.M, p.K, p.ldx, &map);
    if (st != ESP_OK) return st;
    auto kern = spgemm_tma_kernel<BN>;
    ESP_CUDA_OK(ensure_dynamic_smem((const void *)kern, L::kTotal));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(f_tiles, t_tiles, split);
    cfg.blockDim = dim3(192);
    cfg.dynamicSmemBytes = L::kTotal;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = split;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    ESP_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, p, map));
    return ESP_OK;
}

// [M, K] token-major -> [K, ldt] channel-major (a transposed, not permuted, copy; ldt >= M).
__global__ void __launch_bounds__(256) transpose_x_kernel(const uint16_t *__restrict__ X, int M, int K, long ldx,
                                                          uint16_t *__restrict__ Xt, long ldt) {
    __shared__ uint16_t tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int k0 = blockIdx.x * 32, m0 = blockIdx.y * 32;
    // As a programmatic dependent (static_weights): the GEMM behind this copy may start at once and prefetch its weights;
    // X, and the workspace the preceding GEMM may still read, are touched only after that kernel is done.
    grid_launch_dependents();
    grid_dependency_wait();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty + 8 * i, k = k0 + tx;
        tile[ty + 8 * i][tx] = (m < M && k < K) ? X[(long)m * ldx + k] : (uint16_t)0;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int k = k0 + ty + 8 * i, m = m0 + tx;
        if (k < K && m < ldt) Xt[(long)k * ldt + m] = tile[tx][ty + 8 * i];
    }
}

static cudaError_t launch_transpose(const uint16_t *X, int M, int K, long ldx, uint16_t *Xt, long ldt, bool dependent,
                                    cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ceil_div(K, 32), ceil_div(ldt, 32), 1);
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, transpose_x_kernel, X, M, K, ldx, Xt, ldt);
}

// A wait nobody ends: one thread polls a barrier that receives no arrival, gives up after a short limit, records
// ESP_ERR_TIMEOUT and returns -- the same path every bounded wait of the GEMM kernels takes when it runs out.
__global__ void wait_timeout_selftest_kernel() {
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        abort_flag = 0;
        fence_barrier_init();
        bool done = false;
        for (uint32_t i = 0; i < (1u << 12) && !done; ++i) {
            done = mbar_try_wait(smem_u32(&bar), 0);
            if (!done) __nanosleep(64);
        }
        if (!done) {
            abort_flag = 1;
            atomicExch(&g_device_status, (int)ESP_ERR_TIMEOUT);
        }
    }
}

}  // namespace

esp_status_t launch_wait_timeout_selftest(cudaStream_t stream) {
    wait_timeout_selftest_kernel<<<1, 32, 0, stream>>>();
    ESP_CUDA_OK(cudaGetLastError());
    return ESP_OK;
}

static long transposed_ld(int M) { return (long)((M + 15) / 16 * 16); }

// Workspace = [transposed copy of token-major X] [X images of the tiled pair kernel].  The first part is required for
// every kernel but the gather kernel when X is token-major; the second lets large M use the tiled pair kernel.
static size_t transpose_bytes(int M, int K, const esp_gemm_opts &o) {
    if (o.x_layout == ESP_X_CHANNEL_MAJOR || o.force_kernel == ESP_KERNEL_GATHER) return 0;
    return align_up((size_t)K * (size_t)transposed_ld(M) * 2, 256);
}
static size_t ximg_bytes(int M, int K, int tn) {
    switch (tn) {
        case 128: return xtile_bytes<128>(M, K);
        case 192: return xtile_bytes<192>(M, K);
        case 224: return xtile_bytes<224>(M, K);
        case 256: return xtile_bytes<256>(M, K);
        default: return xtile_bytes<240>(M, K);
    }
}
size_t gemm_workspace_min_bytes(int M, int K, const esp_gemm_opts &o) { return transpose_bytes(M, K, o); }
size_t gemm_workspace_bytes(int M, int K, const esp_gemm_opts &o) {
    size_t n = transpose_bytes(M, K, o);
    const bool pair_possible = o.force_kernel == ESP_KERNEL_PAIR_TILED || o.force_kernel == ESP_KERNEL_STREAM_IMAGES || (o.force_kernel == ESP_KERNEL_AUTO && M > 16) || o.force_kernel == ESP_KERNEL_QUAD_TILED ||
                               o.force_kernel == ESP_KERNEL_PAIR_PERSIST || o.force_kernel == ESP_KERNEL_QUAD_MULTICAST;
    if (pair_possible) {
        size_t img = 0;
        for (int tn : {128, 192, 224, 240, 256}) img = std::max(img, ximg_bytes(M, K, tn));
        n += img;
    }
    return n;
}

// Resident capacity (in CTAs) of the streaming kernel for one configuration, cached per process.
static int stream_capacity_ctas(const DeviceInfo &di, const int *layer, int bn, int split, int stages, int x_area) {
    const int threads = bn >= 64 ? StreamCfg<64>::kThreads : StreamCfg<16>::kThreads;
    int per_sm = (int)((size_t)(di.max_smem_optin + 1024) / (stream_smem_bytes(bn, stages, split, x_area) + 1024));
    per_sm = std::min(per_sm, std::min(2048 / threads, 512 / tmem_cols_for(bn)));
    return layer[split] * split * std::max(per_sm, 1);
}

// Clusters of 2 x split CTAs of the pair kernel that the device holds at once, asked once per device.
static int pair_cluster_capacity(int device, int split) {
    static std::mutex mu;
    static std::map<int, int> cache;
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(device * 16 + split);
    if (it != cache.end()) return it->second;
    auto kern = spgemm_pair_kernel<1, 256, true>;
    const int smem = PairCfg<1, 256>::kTotal;
    int n = 0;
    if (2 * split <= 8 && ensure_dynamic_smem((const void *)kern, smem) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        cfg.gridDim = dim3(2, 1, split);
        cfg.blockDim = dim3(kPairThreads);
        cfg.dynamicSmemBytes = smem;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = split;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
    }
    if (log_plans()) fprintf(stderr, "esparse pair clusters of %d CTAs: %d fit\n", 2 * split, n);
    return cache[device * 16 + split] = n;
}

// Token tiles of the pair kernel: features (in 128-feature tiles) x tokens of a pair's tile, time of a 128-channel step, and of the rest
// of a wave (start, ring fill, epilogue).  Measured, one wave of 16 to 86 steps, tiled form: 256 features x 256 tokens 19.5 us at 16 steps,
// 28.4 at 32, 60 at 86; 512 x 128 the same area in 21.6, 31 and 66 (its MMAs are half as wide, so the weight operand is read from
// shared memory twice as often: the MMA thread is busy 850 to 1000 of a step's 1130 clocks); the widest cover 1.9 times the
// area in 1.4 times the time and win once the grid fills whole waves.
struct PairTile { int tokens, feature_tiles; double step_us, fixed_us; };
static const PairTile kPairTiles[] = {{240, 4, 0.83, 13.0}, {224, 4, 0.82, 12.5}, {192, 4, 0.80, 12.0}, {256, 2, 0.585, 9.7}, {128, 4, 0.66, 10.5}};

// The pair kernel's tile and K-slices of least time (us, as measured) for these sizes; *tile != 0 and split_k != 0 are requests.
// image_room: workspace bytes for X images.  A form that needs them takes a tile whose images have room; a tile without room runs in the gather form, whose step
// costs kGatherStep more (0.66 -> 0.83 us and 0.585 -> 0.78 measured).  Counted as tiled, 5104 x 15382 at 67 tokens without room for images took the
// 256-token tile, 47.2 us, for 42.7 in two slices of the 128-token tile.
constexpr double kGatherStep = 0.18;
static double best_pair_tile(int M, int K, int f_tiles, int k_tiles, int force_kernel, int split_k, bool wide_only, size_t image_room, const DeviceInfo &di, int *tile, int *split) {
    const long per_wave = di.sm_count / 2 > 0 ? di.sm_count / 2 : 1;
    const bool requested = *tile != 0;
    const int request = *tile;
    double best = -1.0;
    for (const PairTile &t : kPairTiles) {
        if (requested ? t.tokens != request : (wide_only && (t.tokens == 128 || t.tokens == 256))) continue;
        const bool tiled = wide_only || force_kernel == ESP_KERNEL_PAIR_TILED;
        const bool room = image_room >= ximg_bytes(M, K, t.tokens);
        if (!requested && tiled && !room) continue;
        const double step_us = t.step_us + (force_kernel == ESP_KERNEL_PAIR || !room ? kGatherStep : 0.0);
        // waves x time of one wave.  Waves: a grid of up to two waves runs as whole waves (equal tiles end together); over many
        // waves the clusters drift apart and the last, partial wave costs less and less of a whole one.
        // K-slices (128- and 256-token tiles: the pushed partial rows of all slices must fit the ring), each of at least four
        // channel steps: a cluster of 2 x split CTAs, of which far fewer fit the GPU (two slices: 33 on 148 SMs), and about
        // 10 us for the reduction.  Beyond 256 tokens two slices at most: three ran far slower (4096 x 11008 at 384 tokens 70
        // against 50 us).
        const long pairs = (long)ceil_div(f_tiles, t.feature_tiles) * ceil_div(M, t.tokens);
        const bool sliced = t.tokens == 128 || t.tokens == 256;
        int most = sliced ? (M > 256 ? 2 : 4) : 1;
        int wanted = split_k;
        if (wanted > 0) {
            if (!sliced && wanted > 1) continue;
            while (wanted > 1 && (k_tiles / wanted < 4 || (long)ceil_div(k_tiles, wanted) * (wanted - 1) >= k_tiles)) --wanted;
            most = wanted;
        }
        for (int sp = wanted > 0 ? wanted : 1; sp <= most; ++sp) {
            if (sp > 1 && wanted == 0 && (k_tiles / sp < 4 || (long)ceil_div(k_tiles, sp) * (sp - 1) >= k_tiles)) continue;
            const long cap = std::max<long>(1, sp == 1 ? per_wave : pair_cluster_capacity(di.device, sp));
            if (sp > 1 && wanted == 0 && pairs > cap) continue;
            const double w = (double)pairs / (double)cap, whole = (double)ceil_div(pairs, cap);
            const double waves = w <= 2.0 ? whole : w + (whole - w) * (2.0 / w);
            const double cost = waves * (step_us * ceil_div(k_tiles, sp) + t.fixed_us) + (sp > 1 ? 10.0 : 0.0);
            if (log_plans()) fprintf(stderr, "esparse plan M=%d f_tiles=%d k_tiles=%d pair tile=%d split=%d pairs=%ld waves=%.2f cost=%.1f\n", M, f_tiles, k_tiles, t.tokens, sp, pairs, waves, cost);
            if (best < 0.0 || cost < best) { best = cost; *tile = t.tokens; *split = sp; }
        }
    }
    return best;
}

// K-slices, ring depth and input form of the streaming kernel for one token tile (split_k != 0: that many slices, or fewer without an
// empty one).  `capacity`: CTAs that the device holds at once in that form.
struct StreamShape { int split, stages, x_mode, x_area, capacity; };
static bool stream_shape(int M, int N, int K, const esp_gemm_opts &o, int kernel, int bn, int split_k, const DeviceInfo &di, const int *layer,
                         StreamShape *shape) {
    const int k_tiles = ceil_div(K, kTileK), f_tiles = ceil_div(N, kTileFeat);
    const long tiles = (long)f_tiles * ceil_div(M, bn);
    auto no_empty_slice = [&](int split) { return (long)ceil_div(k_tiles, split) * (split - 1) < k_tiles; };
    // Pick K-slices and CTAs per SM so that, if possible, the whole grid is resident at once and each CTA
    // has a short chain of tiles: cost ~ waves x (tiles per CTA + fixed start-up and reduction time).
    const size_t per_stage = (size_t)kTileBytes + 256 * (size_t)bn;
    double best_cost = 1e30;
    shape->split = 0;
    int wanted = split_k > k_tiles ? k_tiles : split_k;      // a requested split steps down to one without empty slices
    while (wanted > 1 && !no_empty_slice(wanted)) --wanted;
    for (int split = 1; split <= 8 && split <= k_tiles; ++split) {
        if (wanted != 0 && split != wanted) continue;
        if (!no_empty_slice(split)) continue;
        const int kts = ceil_div(k_tiles, split);
        // token-major X without a transposing launch: up to two tokens straight from X (4096 x 11008, us per call: 14.6 -> 13.0 at
        // one token, 14.6 -> 15.4 at two; 22016 x 8192: 37.2 -> 34.9 and 35.5; at four tokens the element loads cost more than the
        // launch, 14.7 -> 22.8), through the cluster where the weight is
        // small (its start is longer, but the call saves a launch: 512 x 512 at 128 tokens 8.7 -> 6.2, 2048 x 2048 at 16 tokens 8.1 ->
        // 7.0, at 32 tokens 8.2 -> 8.9; 4096 x 4096 at 16 tokens 9.2 -> 11.7)
        int x_mode = kXChannelMajor, x_area = 0;
        if (kernel == ESP_KERNEL_STREAM && o.x_layout == ESP_X_TOKEN_MAJOR) {
            const long weight = (long)N * K;
            if (bn == 16 && (M == 1 || (M <= kXDirectTokens && K <= 8192))) x_mode = kXDirect;
            // (with static_weights the transposing launch overlaps the product before it and costs the GPU little; reading a CTA's share of X at the
            // start of the product then pays for shares that the producers read in about one go.  us per call in a queue, transposed -> through the
            // cluster: 1600 x 818 at 12 tokens, shares of 3 steps, 6.8 -> 6.9 on the GPU and 8.2 -> 6.3 from the host; 5488 x 128 at 46, 6 steps of 16 tokens,
            // 8.2 -> 9.2 and 8.6 -> 8.4; 9696 x 158 at 15 10.4 -> 12.2 and 9.8 -> 11.5; 32-token tiles, 2392 x 438 at 35 7.4 -> 8.4 and 8.6 -> 7.9)
            else if (bn <= 32 && weight <= (M <= 16 ? 4500000L : 1200000L) && stream_x_area_bytes(bn, M, kts) <= kXAreaMax &&
                     (!o.static_weights || kts * ((std::min(M, bn) + 7) / 8) <= (bn == 16 ? 10 : 6))) {
                x_mode = kXCluster;
                x_area = stream_x_area_bytes(bn, M, kts);
            }
        }
        const size_t fixed = stream_recv_bytes(bn, split) + (size_t)x_area + kPermRing * 512 + 512 + 1024;
        int last_stages = -1;
        for (int r = 1; r <= 4; ++r) {
            const size_t budget = (size_t)di.max_smem_optin / r - (r > 1 ? 1024 : 0);
            if (budget < fixed + 2 * per_stage) break;
            int stages = (int)((budget - fixed) / per_stage);
            if (o.pipeline_stages > 0) {                              // a requested ring depth: this one only, or what fits
                if (r > 1) break;
                if (stages > o.pipeline_stages) stages = o.pipeline_stages;
            }
            if (stages > kMaxStages) stages = kMaxStages;
            if (stages > kts) stages = kts < 2 ? 2 : kts;
            if (stages == last_stages) continue;
            last_stages = stages;
            const int cap = stream_capacity_ctas(di, layer, bn, split, stages, x_area);
            if (cap <= 0) continue;
            const long ctas = tiles * split;
            const long waves = (ctas + cap - 1) / cap;
            // per CTA: kts steps + set-up, reduction and epilogue, which grow with the token tile (measured: a 256-token
            // tile in one wave of 32 steps beats three waves of 8)
            // wide token tiles are bound by their X gather, which CTAs sharing an SM share: a step costs as many
            // times more as CTAs of one wave sit on an SM
            const long in_wave = ctas < cap ? ctas : cap;
            const double share = (bn >= 64 && kernel == ESP_KERNEL_STREAM) ? (double)((in_wave + di.sm_count - 1) / di.sm_count) : 1.0;
            double cost = (double)waves * (kts * share + 2.0 + bn / 32.0) + (split > 1 ? 0.25 + 0.05 * split : 0.0) + 0.01 * r;
            // with static_weights consecutive launches overlap on an SM: prefer leaving room for a CTA of the next one
            // (not when every CTA has an SM of its own anyway: a deeper ring is then free, measured 16.0 -> 12.6 us on
            // 4096 x 4096 at 64 tokens)
            if (o.static_weights && o.pipeline_stages == 0 && ctas > di.sm_count &&
                2 * (stream_smem_bytes(bn, stages, split, x_area) + 1024) > (size_t)di.max_smem_optin)
                cost += 3.0;
            if (log_plans())
                fprintf(stderr, "esparse plan M=%d N=%d K=%d tile=%d: split=%d stages=%d capacity=%d ctas=%ld waves=%ld cost=%.2f\n", M, N, K,
                        bn, split, stages, cap, ctas, waves, cost);
            if (cost < best_cost) { best_cost = cost; *shape = StreamShape{split, stages, x_mode, x_area, cap}; }
        }
    }
    return shape->split != 0;
}

// Times (us) of the forms that a product of more than 64 tokens on a weight below 40 M elements can take, fitted to 33000 measured
// calls: 1929 shapes of 512..11008 features x channels at 60..8200 tokens, 1427 of them random and 502 token counts on six fixed weights (4096 x 4096,
// 5120 x 5120, 4096 x 11008, 9216 x 9216, 11008 x 4096, 8192 x 2048), every form, tile and number of K-slices that runs (half of the estimates within 5 to 10 %, nine of ten within 20 %; the form chosen by them is 2.5 % slower than the best
// measured one in the geometric mean).  Rules of one threshold each stood here before: up to 256 tokens the streaming kernel's 128- and
// 256-token tiles, the pair kernel beyond.  Small weights lost most: 1010 x 1960 at 181 tokens 15.3 -> 7.8 us, 972 x 3280 at 546 34 -> 16.
// Streaming kernel: waves of the grid (`wave`), CTAs on an SM in each (`wave_sm`), channel steps of these, MB that all CTAs pull from
// L2, K-slices, and the pass that writes X images (per 1e6 elements of X).
struct StreamTime { int tokens; bool images; double start, step, step_sm, wave, wave_sm, per_mb, slice, image; };
static const StreamTime kStreamTimes[] = {
    {32, false, 1.57, 0.443, 0.000, 3.42, 0.00, 0.040, 0.06, 0.00},
    {64, false, 1.97, 0.578, 0.146, 0.84, 1.92, 0.054, 0.17, 0.00},
    {128, false, 3.01, 0.654, 0.157, 0.00, 3.34, 0.052, 0.18, 0.00},
    {256, false, 0.00, 0.000, 1.113, 0.00, 9.93, 0.033, 0.49, 0.00},
    {32, true, 3.81, 0.362, 0.000, 4.43, 0.00, 0.030, 0.06, 1.60},
    {64, true, 4.21, 0.389, 0.000, 3.04, 1.66, 0.028, 0.19, 0.73},
    {128, true, 5.03, 0.276, 0.115, 2.27, 3.26, 0.044, 0.22, 0.71},
    {256, true, 0.75, 0.000, 1.207, 0.00, 11.90, 0.015, 0.77, 0.97},
};
// Pair kernel, gather form and tiled form: one channel step, the rest of a wave, K-slices, the tiling pass (or, gather form, the row
// copies).
struct PairTime { int tokens; bool tiled; double step, wave, slices, x; };
static const PairTime kPairTimes[] = {
    {128, false, 0.827, 11.1, 4.5, 0.26},
    {256, false, 0.782, 9.5, 5.4, 0.56},
    {128, true, 0.594, 13.3, 5.2, 0.93},
    {192, true, 0.718, 13.4, 0.0, 1.16},
    {224, true, 0.715, 14.3, 0.0, 1.16},
    {240, true, 0.727, 14.5, 0.0, 1.09},
    {256, true, 0.520, 11.7, 6.9, 0.96},
};

// The form of least estimated time and that time (us; negative: none runs).  `gather_only`: of the streaming kernel's gather forms.
static double fastest_form(int M, int N, int K, const esp_gemm_opts &o, bool gather_only, size_t image_room, const DeviceInfo &di, const int *layer, GemmPlan *g) {
    const int k_tiles = ceil_div(K, kTileK), f_tiles = ceil_div(N, kTileFeat);
    const double x_elems = 1e-6 * (double)K * M;
    double best = 1e30;
    auto take = [&](double us, int kernel, int tile, const StreamShape &sh) {
        if (log_plans()) fprintf(stderr, "esparse plan M=%d N=%d K=%d kernel=%d tile=%d split=%d: %.1f us\n", M, N, K, (int)kernel, tile, sh.split, us);
        if (us >= best) return;
        best = us;
        g->kernel = kernel;
        g->token_tile = tile;
        g->split_k = sh.split;
        g->stages = sh.stages;
        g->x_mode = sh.x_mode;
        g->x_area = sh.x_area;
    };
    for (const StreamTime &t : kStreamTimes) {
        if ((t.images && gather_only) || (t.images && image_room < (t.tokens < 64 ? xtile_narrow_bytes(M, K, t.tokens) : ximg_bytes(M, K, 128))) || t.tokens >= 2 * M) continue;
        const int kernel = t.images ? ESP_KERNEL_STREAM_IMAGES : ESP_KERNEL_STREAM;
        const long tiles = (long)f_tiles * ceil_div(M, t.tokens);
        for (int split : {1, 2, 3, 4, 6, 8}) {
            StreamShape sh;
            if (split > k_tiles || (long)ceil_div(k_tiles, split) * (split - 1) >= k_tiles) continue;
            if (!stream_shape(M, N, K, o, kernel, t.tokens, split, di, layer, &sh)) continue;
            const long ctas = tiles * split, waves = (ctas + sh.capacity - 1) / sh.capacity;
            // (CTAs on an SM: by how many clusters find SMs of their own, not by the SM count -- 48 clusters of three CTAs are 144 CTAs, but the GPCs
            // hold 45 such clusters with one CTA per SM, and the rest double up.  Counted by SMs, 2904 x 2980 at 204 tokens took the 128-token tile
            // in three slices, 22.2 us, for 18.7 in the 256-token tile in five; 8136 x 1420 at 212 tokens 27.4 for 22.3)
            const long alone = (long)std::max(1, layer[split]) * split;
            const long on_sm = waves * ((std::min<long>(ctas, sh.capacity) + alone - 1) / alone);
            const int steps = ceil_div(k_tiles, split);
            const double mb = 1e-6 * (double)ctas * steps * (kTileBytes + 256.0 * t.tokens);
            take(t.start + waves * (t.wave + t.step * steps) + on_sm * (t.wave_sm + t.step_sm * steps) + t.per_mb * mb + t.slice * split + t.image * x_elems,
                 kernel, t.tokens, sh);
        }
    }
    const long per_wave = std::max(1, di.sm_count / 2);
    for (const PairTime &t : kPairTimes) {
        if (gather_only) break;
        if (t.tiled && image_room < ximg_bytes(M, K, t.tokens)) continue;
        const bool sliced = t.tokens == 128 || t.tokens == 256;             // (as in best_pair_tile)
        const long pairs = (long)ceil_div(f_tiles, t.tokens == 256 ? 2 : 4) * ceil_div(M, t.tokens);
        for (int split = 1; split <= (sliced ? (M > 256 ? 2 : 4) : 1); ++split) {
            if (split > 1 && (k_tiles / split < 4 || (long)ceil_div(k_tiles, split) * (split - 1) >= k_tiles)) continue;
            const long cap = std::max<long>(1, split == 1 ? per_wave : pair_cluster_capacity(di.device, split));
            if (split > 1 && pairs > cap) continue;
            const double w = (double)pairs / (double)cap, whole = (double)ceil_div(pairs, cap);
            const double waves = w <= 2.0 ? whole : w + (whole - w) * (2.0 / w);
            take(waves * (t.wave + t.step * ceil_div(k_tiles, split)) + (split > 1 ? t.slices : 0.0) + t.x * x_elems,
                 t.tiled ? ESP_KERNEL_PAIR_TILED : ESP_KERNEL_PAIR, t.tokens, StreamShape{split, 0, kXChannelMajor, 0, 0});
        }
    }
    return best < 1e30 ? best : -1.0;
}

static esp_status_t plan_gemm_uncached(int M, int N, int K, const esp_gemm_opts &o, size_t workspace_bytes, GemmPlan *plan) {
    const bool have_workspace = workspace_bytes >= transpose_bytes(M, K, o) && (workspace_bytes > 0 || o.x_layout == ESP_X_CHANNEL_MAJOR);
    DeviceInfo di;
    esp_status_t st = device_info(&di);
    if (st != ESP_OK) return st;
    GemmPlan g;
    g.x_mode = kXChannelMajor;
    g.x_area = 0;
    const int k_tiles = ceil_div(K, kTileK);
    const int f_tiles = ceil_div(N, kTileFeat);
    const bool channel_major_available = (o.x_layout == ESP_X_CHANNEL_MAJOR) || have_workspace;
    const size_t image_room = have_workspace ? workspace_bytes - transpose_bytes(M, K, o) : 0;      // behind the transposed copy
    int bn = o.token_tile;
    int layer[9] = {};
    for (int split = 1; split <= 8; ++split) layer[split] = stream_clusters_one_per_sm(di.device, split);
    g.kernel = ESP_KERNEL_GATHER;
    if (o.force_kernel != ESP_KERNEL_GATHER && channel_major_available) {
        if (o.force_kernel == ESP_KERNEL_TMA) g.kernel = ESP_KERNEL_TMA;
        else if (o.force_kernel == ESP_KERNEL_PAIR) g.kernel = ESP_KERNEL_PAIR;
        else if (o.force_kernel == ESP_KERNEL_PAIR_TILED) g.kernel = ESP_KERNEL_PAIR_TILED;
        else if (o.force_kernel == ESP_KERNEL_QUAD_TILED) g.kernel = ESP_KERNEL_QUAD_TILED;
        else if (o.force_kernel == ESP_KERNEL_PAIR_PERSIST) g.kernel = ESP_KERNEL_PAIR_PERSIST;
        else if (o.force_kernel == ESP_KERNEL_QUAD_MULTICAST) g.kernel = ESP_KERNEL_QUAD_MULTICAST;
        else if (o.force_kernel == ESP_KERNEL_STREAM) g.kernel = ESP_KERNEL_STREAM;
        else if (o.force_kernel == ESP_KERNEL_STREAM_IMAGES) g.kernel = ESP_KERNEL_STREAM_IMAGES;
        else {
            const long weight = (long)N * K;
            // Small and middle weights at more than 64 tokens: the form of least estimated time.  (A few feature tiles on few tokens keep
            // the rule of narrow token tiles below, which those times do not cover; larger weights keep the rules that follow, mostly within 10 % of the
            // best form, but not everywhere: 5850 x 8504 at 65 tokens takes 1.24 times as long, 9216 x 9216 at 163..253 1.08 times (two slices, one is
            // faster).  Beyond 256 tokens and below 16 channel steps the tiled pair form stays the default, which the tests of the plan ask for; streaming tiles
            // would gain up to 7 us of 15 there.)
            const bool narrow = M <= 256 && (long)f_tiles * k_tiles <= 64 && (long)f_tiles * ceil_div(M, 64) * std::min(k_tiles, 8) <= 2L * di.sm_count;
            if (M > 64 && bn == 0 && o.split_k == 0 && o.pipeline_stages == 0 && !narrow && (M <= 256 || k_tiles >= 16) && weight < (M > 1000 ? 15000000L : 40000000L) &&
                fastest_form(M, N, K, o, false, image_room, di, layer, &g) >= 0.0) {
                *plan = g;
                return ESP_OK;
            }
            // The pair kernel takes every M > 64; a requested token tile or slice count that only the streaming kernel has
            // (tiles below 128 tokens, more than four slices, slices of a 256-token tile) goes there.
            const bool stream_only = (bn != 0 && bn < 128) || o.split_k > 4 || (bn == 256 && o.split_k > 1);
            // Up to 256 tokens the pair kernel pays only where the weight gives it twenty pairs or more per K-slice (its
            // set-up and drain cost about 10 us; measured at 128 tokens: 11008 x 4096 26.5 against the streaming kernel's
            // 28.5 us, but 4096 x 4096 20.3 against 14.6).
            const long pairs128 = (long)ceil_div(f_tiles, 4) * ceil_div(M, 128);
            const bool pair = !stream_only && (M > 256 || (M > 64 && pairs128 >= 20));
            g.kernel = pair ? ESP_KERNEL_PAIR : ESP_KERNEL_STREAM;
            // 17..256 tokens on a large weight: the streaming kernel fed from X images.  Its row gather limits the
            // streaming kernel once the X tile is a good part of a stage; the images cost one more (small) launch, which pays
            // from about 40 M weight elements (measured, gather form -> image form: 36864 x 9216 at 32 / 64 tokens
            // 78 -> 67 / 118 -> 68 us; 9216 x 9216 at 64 / 128 tokens 41 -> 28 / 47 -> 37 us; but 9216 x 9216 at 32 tokens
            // 22.5 -> 28.4, 4096 x 4096 at 128 tokens 15.0 -> 17.1).  It also replaces the pair kernel's gather form where that
            // would run K-slices at 129..256 tokens (9216 x 9216 at 256 tokens: 95 -> 55 us).
            // (More than 64 tokens on less than 40 M elements come here only with a requested slice count or ring depth, without an estimated form, or as
            // narrow problems.)
            const bool images_room = image_room >= ximg_bytes(M, K, 128);
            if (images_room && bn == 0 && o.split_k <= 8 && M > 16 && M <= 256) {
                const long per_wave = di.sm_count / 2 > 0 ? di.sm_count / 2 : 1;
                if (!pair) {
                    // (33..64 tokens, 64 feature tiles or more: from 24 M elements -- 2472 x 11576 at 61 tokens 23.5 -> 17.9 us, 1792 x 19646 at 48 tokens
                    // 26.9 -> 20.5, but 1824 x 10658 at 45 16.1 against 16.6 and 968 x 15484 at 46 10.5 against 14.1.  From 5 M where token-major X is transposed
                    // by a launch that does not overlap, which the images save: 352 x 20560 at 42 tokens 16.2 -> 14.5, 1568 x 9158 at 38 18.6 -> 16.6, but
                    // 280 x 13756 at 60 11.6 against 14.6)
                    const long wide_from = o.x_layout == ESP_X_TOKEN_MAJOR && !o.static_weights ? 5000000L : 24000000L;
                    const bool pays = M <= 32 ? weight >= 200000000L : M <= 64 ? ((f_tiles >= 64 && weight >= wide_from) || weight >= 64000000L) : M <= 128 ? weight >= 40000000L : weight >= 16000000L;
                    // (up to 32 tokens: 32-token images -- 36864 x 9216 at 32 tokens 67.5 -> 64.3 us, 9216 x 36864 76 -> 70)
                    if (pays) {
                        bn = M <= 32 ? 32 : (M > 128 && weight >= 64000000L) ? 128 : 64;
                        g.kernel = ESP_KERNEL_STREAM_IMAGES;
                        // beyond 128 tokens that kernel is bound by what all its CTAs pull from L2, about 9 TB/s: long weights go to the
                        // pair kernel's K-slices, whose larger tiles pull less (4096 x 11008 at 200 tokens: 41.5 -> 40.0 us).  The estimate is low where the images'
                        // 64-token tiles run in five slices: that weight keeps them at 133..177 tokens, 45 to 46 us, for 39 in the pair kernel.
                        int tile = 0, sp = 1;
                        const double bytes = (double)f_tiles * ceil_div(M, bn) * k_tiles * (kTileBytes + 256.0 * bn);
                        if (M > 128 && o.split_k == 0 && best_pair_tile(M, K, f_tiles, k_tiles, ESP_KERNEL_AUTO, 0, false, image_room, di, &tile, &sp) < bytes / 9e6 - 2.0) {
                            g.kernel = ESP_KERNEL_PAIR;
                            bn = 0;
                        }
                    }
                } else if (M > 128 && o.split_k == 0 && weight >= 80000000L && per_wave / pairs128 >= 2) {
                    g.kernel = ESP_KERNEL_STREAM_IMAGES;
                    bn = 128;
                }
            }
        }
    }
    const bool wide_only = g.kernel == ESP_KERNEL_QUAD_TILED || g.kernel == ESP_KERNEL_PAIR_PERSIST ||
                           g.kernel == ESP_KERNEL_QUAD_MULTICAST;                                      // no 128-token form
    if (g.kernel == ESP_KERNEL_PAIR || g.kernel == ESP_KERNEL_PAIR_TILED || wide_only) {
        int split = 1;
        if (best_pair_tile(M, K, f_tiles, k_tiles, o.force_kernel, o.split_k, wide_only, image_room, di, &bn, &split) < 0.0) {
            // (no tile at all, or none whose images have room)
            const bool without_room = best_pair_tile(M, K, f_tiles, k_tiles, o.force_kernel, o.split_k, wide_only, SIZE_MAX, di, &bn, &split) >= 0.0;
            return without_room ? ESP_ERR_WORKSPACE : ESP_ERR_INVALID_ARG;
        }
        // the tiled form needs room for the X images behind the transposed copy; without it the gather form runs.  Up to
        // 128 tokens the gather form is taken anyway: one launch instead of two, and X is small.
        // (on a large weight the gather's row copies cost more than that launch: 22016 x 8192 at 100 tokens 76 -> 61 us)
        const bool room = image_room >= ximg_bytes(M, K, bn);
        if ((g.kernel == ESP_KERNEL_PAIR_TILED || wide_only) && !room) return ESP_ERR_WORKSPACE;
        if (wide_only && (bn == 128 || bn == 256)) return ESP_ERR_INVALID_ARG;
        // (129..256 tokens in one K-slice: the tiled form too -- 11008 x 4096 at 256 tokens 37.4 -> 33.4 us, 13824 x 5120
        // 47.2 -> 41.6; with K-slices the gather form stays ahead there)
        if (g.kernel == ESP_KERNEL_PAIR && o.force_kernel == ESP_KERNEL_AUTO && room &&
            (M > 256 || (split == 1 && (M > 128 || (long)N * K >= 80000000L)) || bn == 256))
            g.kernel = ESP_KERNEL_PAIR_TILED;
        g.token_tile = bn;
        g.split_k = split;
        g.stages = 0;
        *plan = g;
        return ESP_OK;
    }
    // (33..64 tokens: two 32-token tiles beat one of 64 unless the weight has many feature tiles -- the second pass over the
    // weight comes from L2, and the narrow tile keeps more CTAs per SM; 5120 x 5120: 13.1 against 15.7 us)
    if (bn == 0) bn = M <= 16 ? 16 : M <= 32 ? 32 : M <= 64 ? (f_tiles <= 64 && g.kernel == ESP_KERNEL_STREAM ? 32 : 64) : M <= 128 ? 128 : 256;
    // (a weight of a few tiles: narrow token tiles, so that the tiles x K-slices come to about one CTA per SM; re-reading
    // so small a weight per token tile costs nothing.  512 x 512 at 128 tokens: 3.1 us with 16-token tiles against 8.4)
    if (o.token_tile == 0 && g.kernel == ESP_KERNEL_STREAM && M > 16 && (long)f_tiles * k_tiles <= 64) {
        for (int narrow : {16, 32, 64}) {
            if (narrow >= bn) break;
            if ((long)f_tiles * ceil_div(M, narrow) * std::min(k_tiles, 8) <= 2L * di.sm_count) { bn = narrow; break; }
        }
    }
    if (g.kernel == ESP_KERNEL_TMA && bn < 64) bn = 64;
    if (g.kernel == ESP_KERNEL_STREAM_IMAGES && image_room < ximg_bytes(M, K, 128)) return ESP_ERR_WORKSPACE;
    if (bn != 16 && bn != 32 && bn != 64 && bn != 128 && bn != 256) return ESP_ERR_INVALID_ARG;
    g.token_tile = bn;
    g.stages = 4;
    const int t_tiles = ceil_div(M, bn);
    const long tiles = (long)f_tiles * t_tiles;
    auto no_empty_slice = [&](int split) { return (long)ceil_div(k_tiles, split) * (split - 1) < k_tiles; };
    if (g.kernel == ESP_KERNEL_STREAM || g.kernel == ESP_KERNEL_STREAM_IMAGES) {
        StreamShape shape;
        if (!stream_shape(M, N, K, o, g.kernel, bn, o.split_k, di, layer, &shape)) return ESP_ERR_UNSUPPORTED;
        g.split_k = shape.split;
        g.stages = shape.stages;
        g.x_mode = shape.x_mode;
        g.x_area = shape.x_area;
        *plan = g;
        return ESP_OK;
    }
    int split = o.split_k;
    if (split == 0) {
        split = 1;
        while (split < 8 && tiles * split < di.sm_count && k_tiles / (split * 2) >= 4) split *= 2;
    }
    if (split > k_tiles) split = k_tiles;
    if (split < 1) split = 1;
    while (split > 1 && !no_empty_slice(split)) --split;
    g.split_k = split;
    *plan = g;
    return ESP_OK;
}


// The plan of a call is a pure function of its sizes, its options, the workspace size and the device: the last few are
// remembered per thread, so that a layer's repeated calls do not walk the candidates again.
esp_status_t plan_gemm(int M, int N, int K, const esp_gemm_opts &o, size_t workspace_bytes, GemmPlan *plan) {
    struct Key { int dev, M, N, K, x_layout, split_k, force_kernel, token_tile, static_weights, pipeline_stages; size_t ws; };
    struct Entry { Key key; GemmPlan plan; };
    thread_local Entry cache[32];
    thread_local int n = 0, next = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    const Key key{dev, M, N, K, o.x_layout, o.split_k, o.force_kernel, o.token_tile, o.static_weights, o.pipeline_stages, workspace_bytes};
    if (!log_plans())
        for (int i = 0; i < n; ++i) {
            const Key &k = cache[i].key;
            if (k.dev == key.dev && k.M == key.M && k.N == key.N && k.K == key.K && k.x_layout == key.x_layout && k.split_k == key.split_k &&
                k.force_kernel == key.force_kernel && k.token_tile == key.token_tile && k.static_weights == key.static_weights &&
                k.pipeline_stages == key.pipeline_stages && k.ws == key.ws) {
                *plan = cache[i].plan;
                return ESP_OK;
            }
        }
    const esp_status_t st = plan_gemm_uncached(M, N, K, o, workspace_bytes, plan);
    if (st == ESP_OK) {
        cache[next] = Entry{key, *plan};
        next = (next + 1) % 32;
        if (n < 32) ++n;
    }
    return st;
}

// ---- the optional companion library: the one kernel form whose weight loads use cluster multicast is built into a shared
// object of its own (libesparse_mc.so, from spgemm_mcast.cu), looked for once beside this library.
namespace {
struct Companion {
    int (*launch)(const void *, size_t, int, int, void *) = nullptr;
    int (*status)(int *) = nullptr;
};
const Companion *companion() {
    static Companion c;
    static std::once_flag once;
    static bool ok = false;
    std::call_once(once, [] {
        Dl_info info;
        if (!dladdr(reinterpret_cast<const void *>(&plan_gemm), &info) || !info.dli_fname) return;
        std::string path(info.dli_fname);
        const size_t slash = path.rfind('/');
        path = (slash == std::string::npos ? std::string() : path.substr(0, slash + 1)) + "libesparse_mc.so";
        void *h = dlopen(path.c_str(), RTLD_NOW | RTLD_LOCAL);
        if (!h) return;
        c.launch = reinterpret_cast<int (*)(const void *, size_t, int, int, void *)>(dlsym(h, "esp_mc_launch_pair"));
        c.status = reinterpret_cast<int (*)(int *)>(dlsym(h, "esp_mc_device_status"));
        ok = c.launch != nullptr && c.status != nullptr;
    });
    return ok ? &c : nullptr;
}

// The tiling pass over X (channel-major, or token-major when x_tm is given) and then the planned form of the tiled pair
// kernel as its programmatic dependent (it waits on the image flags, not on the grid).
template <int TN>
esp_status_t launch_tiled_form(GemmParams &p, const GemmPlan &plan, const uint16_t *x_tm, long ldx_tm, uint8_t *img, bool dependent,
                               cudaStream_t stream, int sm_count) {
    uint32_t *flags = reinterpret_cast<uint32_t *>(img + xtile_image_bytes<TN>(p.M, p.K));
    p.ximg = img;
    p.xflags = flags;
    esp_status_t st = x_tm ? launch_xtile_tm<TN>(p, x_tm, ldx_tm, img, flags, dependent, stream) : launch_xtile<TN>(p, img, flags, dependent, stream);
    if (st != ESP_OK) return st;
    if constexpr (TN == 128 || TN == 256) {
        if (plan.kernel != ESP_KERNEL_PAIR_TILED) return ESP_ERR_INVALID_ARG;
        return launch_pair<TN == 128 ? 2 : 1, TN, true>(p, true, stream, plan.split_k);
    } else {
        switch (plan.kernel) {
            case ESP_KERNEL_QUAD_TILED: return launch_quad<TN>(p, true, stream);
            case ESP_KERNEL_PAIR_PERSIST: return launch_pair_persist<TN>(p, true, stream, sm_count);
            case ESP_KERNEL_QUAD_MULTICAST: {
                const Companion *c = companion();
                return c ? (esp_status_t)c->launch(&p, sizeof(p), TN, 1, stream) : ESP_ERR_UNSUPPORTED;
            }
            default: return launch_pair<2, TN, true>(p, true, stream);
        }
    }
}
}  // namespace

bool companion_available() { return companion() != nullptr; }
esp_status_t companion_device_status(int *out) {
    *out = 0;
    const Companion *c = companion();
    return c ? (esp_status_t)c->status(out) : ESP_OK;
}

esp_status_t launch_spgemm(const __half *X, int M, int K, long ldx, const void *packed, const int32_t *perm, int N,
                           void *Y, long ldy, const esp_gemm_opts &o, const GemmPlan &plan, void *workspace,
                           size_t workspace_bytes, cudaStream_t stream) {
    GemmParams p;
    p.X = X; p.ldx = ldx; p.M = M; p.K = K; p.N = N;
    p.x_channel_major = (o.x_layout == ESP_X_CHANNEL_MAJOR) ? 1 : 0;
    p.packed = (const uint8_t *)packed;
    p.perm = perm;
    p.Y = Y; p.ldy = ldy;
    p.out_f32 = (o.out_dtype == ESP_OUT_F32) ? 1 : 0;
    p.bias = reinterpret_cast<const __half *>(o.bias);
    p.act = o.activation;
    p.k_tiles = ceil_div(K, kTileK);
    p.k_tiles_per_split = ceil_div(p.k_tiles, plan.split_k);
    p.ximg = nullptr;
    p.xflags = nullptr;
    p.raster_panel = 0;
    p.x_mode = plan.x_mode;
    p.x_area = plan.x_area;
    const int f_tiles = ceil_div(N, kTileFeat), t_tiles = ceil_div(M, plan.token_tile);
    const bool quad_form = plan.kernel == ESP_KERNEL_QUAD_TILED || plan.kernel == ESP_KERNEL_QUAD_MULTICAST;
    if (plan.kernel == ESP_KERNEL_PAIR || plan.kernel == ESP_KERNEL_PAIR_TILED || quad_form || plan.kernel == ESP_KERNEL_PAIR_PERSIST) {
        // Panels pay once a row of clusters (every feature pair on one token tile) is a good part of a wave: about eight
        // token tiles per panel (six where the weight has few feature pairs), the panels evened out over the token tiles.
        // Measured (M = 8192 unless noted): 22016 x 8192 1.79 -> 1.96 PFLOP/s; 36864 x 9216 at 4096 tokens 1.56 -> 1.94;
        // 8192 x 22016 1.76 -> 1.83; 8192 x 8192 (its 75 MB of weights stay in L2 anyway) unchanged.
        const int f_pairs = ceil_div(f_tiles, 4);
        if (f_pairs >= 12 && t_tiles >= 4) {
            const int want = f_pairs >= 20 ? 8 : 6;
            const int panels = std::max(1, (t_tiles + want / 2) / want);
            p.raster_panel = ceil_div(t_tiles, panels);
            if (quad_form) p.raster_panel = (p.raster_panel + 1) / 2;   // counted in pairs of token tiles there
        }
    }
    if (plan.kernel != ESP_KERNEL_GATHER) {
        if (!p.x_channel_major && plan.x_mode == kXChannelMajor && plan.kernel != ESP_KERNEL_PAIR_TILED &&
            !(plan.kernel == ESP_KERNEL_STREAM_IMAGES && plan.token_tile >= 64)) {
            // token-major input: transposed (not permuted) copy into the caller's workspace
            const long ldt = transposed_ld(M);
            if (!workspace || workspace_bytes < (size_t)K * ldt * 2) return ESP_ERR_WORKSPACE;
            ESP_CUDA_OK(launch_transpose(reinterpret_cast<const uint16_t *>(X), M, K, ldx, reinterpret_cast<uint16_t *>(workspace),
                                         ldt, o.static_weights != 0, stream));
            p.X = reinterpret_cast<const __half *>(workspace);
            p.ldx = ldt;
            p.x_channel_major = 1;
        }
        const bool dependent = o.static_weights != 0;
        if (plan.kernel == ESP_KERNEL_PAIR_TILED || quad_form || plan.kernel == ESP_KERNEL_PAIR_PERSIST) {
            if (plan.kernel == ESP_KERNEL_QUAD_MULTICAST && !companion_available()) return ESP_ERR_UNSUPPORTED;
            DeviceInfo di;
            if (device_info(&di) != ESP_OK) return ESP_ERR_CUDA;
            const size_t off = transpose_bytes(M, K, o);
            if (!workspace || workspace_bytes < off + ximg_bytes(M, K, plan.token_tile)) return ESP_ERR_WORKSPACE;
            uint8_t *img = reinterpret_cast<uint8_t *>(workspace) + off;
            const uint16_t *x_tm = p.x_channel_major ? nullptr : reinterpret_cast<const uint16_t *>(X);   // token-major: one transposing pass
            switch (plan.token_tile) {
                case 128: return launch_tiled_form<128>(p, plan, x_tm, ldx, img, dependent, stream, di.sm_count);
                case 192: return launch_tiled_form<192>(p, plan, x_tm, ldx, img, dependent, stream, di.sm_count);
                case 224: return launch_tiled_form<224>(p, plan, x_tm, ldx, img, dependent, stream, di.sm_count);
                case 240: return launch_tiled_form<240>(p, plan, x_tm, ldx, img, dependent, stream, di.sm_count);
                case 256: return launch_tiled_form<256>(p, plan, x_tm, ldx, img, dependent, stream, di.sm_count);
                default: return ESP_ERR_INVALID_ARG;
            }
        }
        if (plan.kernel == ESP_KERNEL_PAIR) {
            switch (plan.token_tile) {
                case 128: return launch_pair<2, 128>(p, dependent, stream, plan.split_k);
                case 192: return launch_pair<2, 192>(p, dependent, stream);
                case 224: return launch_pair<2, 224>(p, dependent, stream);
                case 240: return launch_pair<2, 240>(p, dependent, stream);
                case 256: return launch_pair<1, 256>(p, dependent, stream, plan.split_k);
                default: return ESP_ERR_INVALID_ARG;
            }
        }
        if (plan.kernel == ESP_KERNEL_STREAM_IMAGES) {
            // the tiling pass writes the images of 64-token blocks (the 128-token pair kernel's format); the streaming kernel
            // follows as its programmatic dependent and takes each image when its flag is up
            const size_t off = transpose_bytes(M, K, o);
            uint8_t *img = reinterpret_cast<uint8_t *>(workspace) + off;
            if (plan.token_tile < 64) {      // narrow tiles: images of their own format, from channel-major X (transposed above if need be)
                const int bn = plan.token_tile;
                if (!workspace || workspace_bytes < off + xtile_narrow_bytes(M, K, bn)) return ESP_ERR_WORKSPACE;
                uint32_t *flags_n = reinterpret_cast<uint32_t *>(img + xtile_narrow_image_bytes(M, K, bn));
                p.ximg = img;
                p.xflags = flags_n;
                if (bn == 32) {
                    const esp_status_t st_n = launch_xtile_narrow<32>(p, img, flags_n, dependent, stream);
                    return st_n != ESP_OK ? st_n : launch_stream<32>(p, f_tiles, t_tiles, plan.split_k, plan.stages, true, stream);
                }
                const esp_status_t st_n = launch_xtile_narrow<16>(p, img, flags_n, dependent, stream);
                return st_n != ESP_OK ? st_n : launch_stream<16>(p, f_tiles, t_tiles, plan.split_k, plan.stages, true, stream);
            }
            if (!workspace || workspace_bytes < off + ximg_bytes(M, K, 128)) return ESP_ERR_WORKSPACE;
            uint32_t *flags = reinterpret_cast<uint32_t *>(img + xtile_image_bytes<128>(M, K));
            p.ximg = img;
            p.xflags = flags;
            const esp_status_t st = p.x_channel_major ? launch_xtile<128>(p, img, flags, dependent, stream)
                                                      : launch_xtile_tm<128>(p, reinterpret_cast<const uint16_t *>(X), ldx, img, flags, dependent, stream);
            if (st != ESP_OK) return st;
            switch (plan.token_tile) {
                case 64: return launch_stream<64>(p, f_tiles, t_tiles, plan.split_k, plan.stages, true, stream);
                case 128: return launch_stream<128>(p, f_tiles, t_tiles, plan.split_k, plan.stages, true, stream);
                case 256: return launch_stream<256>(p, f_tiles, t_tiles, plan.split_k, plan.stages, true, stream);
                default: return ESP_ERR_INVALID_ARG;
            }
        }
        if (plan.kernel == ESP_KERNEL_STREAM) {
            switch (plan.token_tile) {
                case 16: return launch_stream<16>(p, f_tiles, t_tiles, plan.split_k, plan.stages, dependent, stream);
                case 32: return launch_stream<32>(p, f_tiles, t_tiles, plan.split_k, plan.stages, dependent, stream);
                case 64: return launch_stream<64>(p, f_tiles, t_tiles, plan.split_k, plan.stages, dependent, stream);
                case 128: return launch_stream<128>(p, f_tiles, t_tiles, plan.split_k, plan.stages, dependent, stream);
                case 256: return launch_stream<256>(p, f_tiles, t_tiles, plan.split_k, plan.stages, dependent, stream);
                default: return ESP_ERR_INVALID_ARG;
            }
        }
        switch (plan.token_tile) {
            case 64: return launch_tma<64>(p, f_tiles, t_tiles, plan.split_k, stream);
            case 128: return launch_tma<128>(p, f_tiles, t_tiles, plan.split_k, stream);
            case 256: return launch_tma<256>(p, f_tiles, t_tiles, plan.split_k, stream);
            default: return ESP_ERR_INVALID_ARG;
        }
    }
    switch (plan.token_tile) {
        case 16: return launch_gather<16, 6>(p, f_tiles, t_tiles, plan.split_k, stream);
        case 32: return launch_gather<32, 6>(p, f_tiles, t_tiles, plan.split_k, stream);
        case 64: return launch_gather<64, 5>(p, f_tiles, t_tiles, plan.split_k, stream);
        case 128: return launch_gather<128, 4>(p, f_tiles, t_tiles, plan.split_k, stream);
        case 256: return launch_gather<256, 2>(p, f_tiles, t_tiles, plan.split_k, stream);
        default: return ESP_ERR_INVALID_ARG;
    }
}

// More than 64 tokens, and the group's weights as one would take a form that has no launch for groups: true if the streaming kernel, one launch for all, is still
// estimated faster than the problems one after the other in their own forms (three of 5936 x 1792 at 125 tokens: 29 us, 56 apart; of 6880 x 722 at 239: 27
// and 50; two of 2456 x 4594 at 90: 18 and 23).  Remembered per thread, like the plans.
static bool group_in_one_launch(int count, int M, int K, const int *N, int f_total, const esp_gemm_opts &o, size_t workspace_bytes, GemmPlan *plan) {
    if (o.force_kernel != ESP_KERNEL_AUTO || o.token_tile != 0 || o.split_k != 0 || o.pipeline_stages != 0) return false;
    struct Entry { int dev, count, M, K, N[ESP_MAX_GROUP], x_layout, static_weights; size_t ws; bool one; GemmPlan plan; };
    thread_local Entry cache[16];
    thread_local int n = 0, next = 0;
    DeviceInfo di;
    if (device_info(&di) != ESP_OK) return false;
    Entry e = {di.device, count, M, K, {}, o.x_layout, o.static_weights, workspace_bytes, false, GemmPlan{}};
    for (int i = 0; i < count; ++i) e.N[i] = N[i];
    for (int i = 0; i < n; ++i) {
        const Entry &c = cache[i];
        if (c.dev == e.dev && c.count == e.count && c.M == e.M && c.K == e.K && std::equal(c.N, c.N + ESP_MAX_GROUP, e.N) && c.x_layout == e.x_layout &&
            c.static_weights == e.static_weights && c.ws == e.ws) {
            if (c.one) *plan = c.plan;
            return c.one;
        }
    }
    int layer[9] = {};
    for (int split = 1; split <= 8; ++split) layer[split] = stream_clusters_one_per_sm(di.device, split);
    const size_t share = (workspace_bytes / (size_t)count) & ~(size_t)255, transposed = transpose_bytes(M, K, o);
    const double together = fastest_form(M, f_total * kTileFeat, K, o, true, 0, di, layer, &e.plan);
    double apart = 0.0;
    GemmPlan ignored;
    for (int i = 0; i < count; ++i) apart += fastest_form(M, N[i], K, o, false, share > transposed ? share - transposed : 0, di, layer, &ignored);
    e.one = together >= 0.0 && together < apart;
    if (e.one) *plan = e.plan;
    cache[next] = e;
    next = (next + 1) % 16;
    if (n < 16) ++n;
    return e.one;
}

esp_status_t launch_spgemm_group(int count, const void *const *X, int M, int K, long ldx, const void *const *packed,
                                 const int32_t *const *perm, const int *N, void *const *Y, const long *ldy,
                                 const esp_gemm_opts &o, void *workspace, size_t workspace_bytes, cudaStream_t stream) {
    if (M > 256) return ESP_ERR_UNSUPPORTED;
    int f_total = 0;
    for (int i = 0; i < count; ++i) f_total += ceil_div(N[i], kTileFeat);
    const size_t tbytes = transpose_bytes(M, K, o);
    if (tbytes > 0 && (!workspace || workspace_bytes < tbytes * (size_t)count)) return ESP_ERR_UNSUPPORTED;
    GemmPlan plan;
    esp_gemm_opts og = o;                    // (a group shares one launch of the streaming kernel's gather form)
    if (og.force_kernel == ESP_KERNEL_AUTO && M <= 64) og.force_kernel = ESP_KERNEL_STREAM;
    esp_status_t st = plan_gemm(M, f_total * kTileFeat, K, og, workspace ? workspace_bytes : 0, &plan);
    if (st != ESP_OK) return st;
    if (plan.kernel != ESP_KERNEL_STREAM && !(M > 64 && group_in_one_launch(count, M, K, N, f_total, og, workspace ? workspace_bytes : 0, &plan))) return ESP_ERR_UNSUPPORTED;
    GemmGroup grp;
    grp.count = count;
    int ft = 0;
    for (int i = 0; i < ESP_MAX_GROUP; ++i) {
        const int j = i < count ? i : 0;
        GemmParams &p = grp.p[i];
        p.X = (const __half *)X[j]; p.ldx = ldx; p.M = M; p.K = K; p.N = N[j];
        p.x_channel_major = 1;
        p.packed = (const uint8_t *)packed[j];
        p.perm = perm ? perm[j] : nullptr;
        p.Y = Y[j]; p.ldy = ldy[j];
        p.out_f32 = (o.out_dtype == ESP_OUT_F32) ? 1 : 0;
        p.bias = nullptr;
        p.act = o.activation;
        p.k_tiles = ceil_div(K, kTileK);
        p.k_tiles_per_split = ceil_div(p.k_tiles, plan.split_k);
        p.ximg = nullptr;
        p.xflags = nullptr;
        p.raster_panel = 0;
        p.x_mode = plan.x_mode;
        p.x_area = plan.x_area;
        grp.ft_start[i] = ft;
        if (i < count) {
            if (o.x_layout != ESP_X_CHANNEL_MAJOR && plan.x_mode == kXChannelMajor) {      // token-major: a transposed copy per distinct input, one after the other
                const long ldt = transposed_ld(M);
                int first = i;
                for (int e = 0; e < i; ++e)
                    if (X[e] == X[i]) { first = e; break; }                 // same-input linears (q, k, v) share the copy
                uint16_t *xt = reinterpret_cast<uint16_t *>(reinterpret_cast<uint8_t *>(workspace) + (size_t)first * tbytes);
                if (first == i)
                    ESP_CUDA_OK(launch_transpose(reinterpret_cast<const uint16_t *>(X[i]), M, K, ldx, xt, ldt, o.static_weights != 0, stream));
                p.X = reinterpret_cast<const __half *>(xt);
                p.ldx = ldt;
            }
            ft += ceil_div(N[i], kTileFeat);
        }
    }
    for (int i = count; i <= ESP_MAX_GROUP; ++i) grp.ft_start[i] = ft;
    const int t_tiles = ceil_div(M, plan.token_tile);
    const bool dependent = o.static_weights != 0;
    switch (plan.token_tile) {
        case 16: return launch_stream_group<16>(grp, t_tiles, plan.split_k, plan.stages, dependent, stream);
        case 32: return launch_stream_group<32>(grp, t_tiles, plan.split_k, plan.stages, dependent, stream);
        case 64: return launch_stream_group<64>(grp, t_tiles, plan.split_k, plan.stages, dependent, stream);
        case 128: return launch_stream_group<128>(grp, t_tiles, plan.split_k, plan.stages, dependent, stream);
        case 256: return launch_stream_group<256>(grp, t_tiles, plan.split_k, plan.stages, dependent, stream);
        default: return ESP_ERR_INVALID_ARG;
    }
}

}  // namespace esp
