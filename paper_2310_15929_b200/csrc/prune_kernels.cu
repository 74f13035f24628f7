// Producer side of the E-Sparse hot path: channel statistics (Eq. 1, Eq. 2), score (Eq. 3), global
// naive shuffle, local block shuffle (Algorithm 1, Eq. 5), 2-of-4 selection and compression.
//
// All of these stream fp16 matrices once or twice; they are bound by HBM and by instruction issue, the block shuffle by
// instruction issue and, on short weights, by the latency of a swap.  Every discrete decision is the one that fp64 quantities with explicit round-to-nearest
// multiplies/adds (no FMA contraction) give, over sums of |W| taken exactly in 64-bit integers of 2^-24, so results do not depend on the order in which
// threads visit rows.  The block shuffle need not form those sums for most of its swaps: fp32 sums with proven bounds tell which pair they would choose
// (lbs_bounds.cuh), and where the bounds leave a choice the pairs in question are evaluated exactly.
#include "esp_common.cuh"

#include <math.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <type_traits>

#include "spgemm_device.cuh"

namespace esp {

namespace {

__device__ __forceinline__ double half_bits_abs_to_double(uint16_t h) {
    return (double)__half2float(__ushort_as_half((unsigned short)(h & 0x7FFFu)));
}

// |h| as an integer multiple of 2^-24 (exact for every finite fp16).
__device__ __forceinline__ long long half_bits_abs_fixed(uint16_t h) {
    int e = (h >> 10) & 31;
    long long m = h & 1023;
    return e == 0 ? m : ((1024 + m) << (e - 1));
}

// Two fp32 values per register pair and instruction.
__device__ __forceinline__ uint64_t f32x2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// A launch that may be set up while the preceding kernel runs: the kernels launched this way wait for it (griddepcontrol.wait) before
// their first access to memory, so stream order holds; what they save is the gap between two launches.  `cluster`: CTAs per cluster
// along y.
template <typename... Params, typename... Args>
inline cudaError_t launch_overlapped(void (*kern)(Params...), dim3 grid, int cluster, int threads, size_t smem, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = cluster;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}

// --------------------------------------------------------------------------------------------------
// K1: per-channel sum of squares (fp64), min and max.   Eq. 2 / range of Eq. 1.
// grid (ceil(C/64), splits of the tokens), cluster (1, splits), block 256 = 8 channel-vectors of 8 x 32 token lanes.  32768 x 4096 (268 MB) runs at
// 4.7 TB/s, 0.72 of the copy rate, with the pipe of the conversions to fp64 60 % busy; a chunk of 2048 x 8192 (34 MB) in 11 to 14 us, half of it start,
// merge and drain.  The splits of a column block are one cluster: their partial results meet in distributed shared memory, added in split
// order -- deterministic, without partial arrays in HBM and without a second kernel (which, with one thread per channel, took 8 us
// for 8 splits of 8192 channels and 37 us for 64 of 4096) or a last-CTA tail (8 us).  2048 x 8192: 13.5 + 8.5 -> 14 us.
// --------------------------------------------------------------------------------------------------
struct ColStatsOut {
    double *sumsq;                           // running sum of squares (streaming calibration), or NULL:
    double *norm;                            // the norm of this call's tokens
    double *lo, *hi;                         // running (sumsq != NULL) or this call's range
};
__device__ __forceinline__ double ld_cluster_f64(const double *local, uint32_t rank) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(map_to_rank(smem_u32(local), rank)) : "memory");
    return v;
}
constexpr int kColAhead = 8;                                              // rows each thread keeps in flight
constexpr int kColSmem = (kColAhead + 1) * 256 * 16;                      // the threads' load rings
__global__ void __launch_bounds__(256) colstats_kernel(const __half *__restrict__ X, int T, int C, long ldx, int rows_per_split,
                                                       const ColStatsOut out) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ double s_acc[8][64], s_sum[64];
    __shared__ float s_mn[8][64], s_mx[8][64], s_lo[64], s_hi[64];
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const int c0 = (blockIdx.x * 8 + tx) * 8;
    const int splits = gridDim.y, rank = blockIdx.y;
    const int r_begin = rank * rows_per_split;
    const int r_end = min(T, r_begin + rows_per_split);
    double acc[8];
    __half2 mn[4], mx[4];                                     // (two channels per instruction; NaNs are passed over)
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        mn[k] = __half2half2(__ushort_as_half((unsigned short)0x7C00));
        mx[k] = __half2half2(__ushort_as_half((unsigned short)0xFC00));
    }
    grid_dependency_wait();
    grid_launch_dependents();
    // the channel that this thread finishes (if any), and the state it adds to
    const int c = blockIdx.x * 64 + tid;
    const bool mine = tid < 64 && tid % splits == rank && c < C;
    double run_sumsq = 0.0, run_lo = INFINITY, run_hi = -INFINITY;
    if (mine && out.sumsq) { run_sumsq = out.sumsq[c]; run_lo = out.lo[c]; run_hi = out.hi[c]; }
    if (c0 < C) {
        auto add_row = [&](const uint4 &v) {
            const __half2 *h = reinterpret_cast<const __half2 *>(&v);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 f = __half22float2(h[k]);
                acc[2 * k] = __dadd_rn(acc[2 * k], (double)(f.x * f.x));   // f*f is exact in fp32 (22-bit product)
                acc[2 * k + 1] = __dadd_rn(acc[2 * k + 1], (double)(f.y * f.y));
                mn[k] = __hmin2(mn[k], h[k]);
                mx[k] = __hmax2(mx[k], h[k]);
            }
        };
        // This thread's rows are r_begin + ty + 32 i, i < n; kColAhead of its 16-byte pieces are kept in flight through a private slot
        // ring in shared memory (asynchronous copies, one group per row; one slot more than rows in flight, so the slot being
        // refilled is the one read an iteration ago) -- the registers leave no room for that many rows.
        const int n = (r_end - r_begin - ty + 31) / 32;
        const __half *xcol = X + (long)(r_begin + ty) * ldx + c0;
        uint4 *ring = reinterpret_cast<uint4 *>(s_dyn) + tid;             // slot j of this thread: ring[256 * j]
        const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
        int wr = 0;
        auto fetch = [&](int i) {
            if (i < n)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ring_s + (uint32_t)(wr * 4096)), "l"(xcol + (long)i * 32 * ldx)
                             : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");          // (an empty group past the end keeps the count in step)
            wr = wr == kColAhead ? 0 : wr + 1;
        };
#pragma unroll
        for (int i = 0; i < kColAhead; ++i) fetch(i);
        int rd = 0;
        for (int i = 0; i < n; ++i) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kColAhead - 1) : "memory");
            const uint4 v = ring[256 * rd];
            rd = rd == kColAhead ? 0 : rd + 1;
            fetch(i + kColAhead);
            add_row(v);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    // the four token lanes of a warp, the eight warps, the CTAs of the cluster: each in a fixed order
#pragma unroll
    for (int o = 8; o <= 16; o <<= 1) {
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k] = __dadd_rn(acc[k], __shfl_xor_sync(0xFFFFFFFFu, acc[k], o));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            mn[k] = __hmin2(mn[k], __shfl_xor_sync(0xFFFFFFFFu, mn[k], o));
            mx[k] = __hmax2(mx[k], __shfl_xor_sync(0xFFFFFFFFu, mx[k], o));
        }
    }
    if ((tid & 31) < 8) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            s_acc[tid >> 5][tx * 8 + k] = acc[k];
            s_mn[tid >> 5][tx * 8 + k] = __half2float(k & 1 ? __high2half(mn[k >> 1]) : __low2half(mn[k >> 1]));
            s_mx[tid >> 5][tx * 8 + k] = __half2float(k & 1 ? __high2half(mx[k >> 1]) : __low2half(mx[k >> 1]));
        }
    }
    __syncthreads();
    if (tid < 64) {
        double a = 0.0;
        float lo = INFINITY, hi = -INFINITY;
#pragma unroll
        for (int y = 0; y < 8; ++y) {
            a = __dadd_rn(a, s_acc[y][tid]);
            lo = fminf(lo, s_mn[y][tid]);
            hi = fmaxf(hi, s_mx[y][tid]);
        }
        s_sum[tid] = a;
        s_lo[tid] = lo;
        s_hi[tid] = hi;
    }
    cluster_sync_all();
    if (mine) {
        double a = 0.0;
        float lo = INFINITY, hi = -INFINITY;
#pragma unroll 8
        for (int r = 0; r < splits; ++r) {
            a = __dadd_rn(a, ld_cluster_f64(&s_sum[tid], (uint32_t)r));
            lo = fminf(lo, ld_dsmem_f32(smem_u32(&s_lo[tid]), (uint32_t)r));
            hi = fmaxf(hi, ld_dsmem_f32(smem_u32(&s_hi[tid]), (uint32_t)r));
        }
        if (out.sumsq) {                     // one chunk folded into the running state (chunk order = call order)
            out.sumsq[c] = __dadd_rn(run_sumsq, a);
            out.lo[c] = fmin(run_lo, (double)lo);
            out.hi[c] = fmax(run_hi, (double)hi);
        } else {
            out.norm[c] = sqrt(a);
            out.lo[c] = (double)lo;
            out.hi[c] = (double)hi;
        }
    }
    cluster_sync_all();                      // the partial results of this CTA have been read
}

// Token splits of the statistics pass: up to four CTAs per SM (that many fit, and a second wave of a few would double the time), 64
// token rows each at least, one cluster (eight CTAs).
inline esp_status_t launch_colstats(const __half *X, int T, int C, long ldx, const ColStatsOut &out, int sm_count, cudaStream_t stream) {
    const int cols = ceil_div(C, 64);
    const int splits = std::max(1, std::min({8, 4 * sm_count / cols, ceil_div(T, 64)}));
    ESP_CUDA_OK(launch_overlapped(colstats_kernel, dim3(cols, splits), splits, 256, kColSmem, stream, X, T, C, ldx, ceil_div(T, splits), out));
    return ESP_OK;
}

// The layer-wide bin range: every channel's [lo, hi] replaced by the minimum and maximum over all channels (one CTA).
__global__ void __launch_bounds__(1024) global_range_kernel(int C, double *__restrict__ lo, double *__restrict__ hi) {
    __shared__ double s_lo[32], s_hi[32];
    double mn = INFINITY, mx = -INFINITY;
    for (int c = threadIdx.x; c < C; c += 1024) { mn = fmin(mn, lo[c]); mx = fmax(mx, hi[c]); }
    for (int o = 16; o > 0; o >>= 1) {
        mn = fmin(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
        mx = fmax(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    }
    if ((threadIdx.x & 31) == 0) { s_lo[threadIdx.x >> 5] = mn; s_hi[threadIdx.x >> 5] = mx; }
    __syncthreads();
    mn = s_lo[0]; mx = s_hi[0];
    for (int w = 1; w < 32; ++w) { mn = fmin(mn, s_lo[w]); mx = fmax(mx, s_hi[w]); }
    __syncthreads();
    for (int c = threadIdx.x; c < C; c += 1024) { lo[c] = mn; hi[c] = mx; }
}

__global__ void calib_reset_kernel(int C, int bins, double *sumsq, double *lo, double *hi, unsigned int *counts) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < C) { sumsq[i] = 0.0; lo[i] = INFINITY; hi[i] = -INFINITY; }
    if (i < (long)C * bins) counts[i] = 0u;
}

// --------------------------------------------------------------------------------------------------
// K2: per-channel histogram with K equal-width bins on [lo_c, hi_c] (Eq. 1's bins), exact integer counts.
// bin = min(K-1, floor((x - lo) * K / (hi - lo))) in fp64: the numerator is exact and the quotient is
// correctly rounded, which yields the exact bin for fp16 data.
// grid (ceil(C/64), splits), block 256 = 8 channel-vectors of 8 x 32 token lanes; counters in shared memory.
// --------------------------------------------------------------------------------------------------
// The exact bin of one element (fp64), for the few elements the fp32 estimate cannot decide.  Kept out of line so that the
// streaming loop carries none of its operands in registers: the channel's range is re-read (from L1) when needed.
__device__ __noinline__ int histogram_exact_bin(float xf, int c, int bins, const double *__restrict__ lo,
                                                const double *__restrict__ hi) {
    const double l = lo[c];
    const double rng = __dsub_rn(hi[c], l);
    if (!(rng > 0.0)) return 0;                                          // a constant channel: everything in bin 0
    const double q = __ddiv_rn(__dmul_rn(__dsub_rn((double)xf, l), (double)bins), rng);
    return max(0, min(bins - 1, (int)floor(q)));                         // (the clamp at 0 only keeps a NaN in bounds)
}

// Counters in shared memory: [k = channel within the thread's eight][bin][tx = the thread's channel group][replica].
// The 32 lanes of a warp are 8 channel groups x 4 token rows, and one instruction counts the same k in all of them, so a
// lane's bank is (bin * 8 + tx) * R + replica: lanes of different channel groups never meet in a bank, and the four lanes
// of a group meet only through the low bits of their bins.  R = 4 gives each of them a counter row of its own (no conflict
// at all), R = 2 one per two, R = 1 none (expected 1.0 / 1.5 / 2.1 passes per counting instruction; the plain
// [channel][bin] layout needed 3.3).  R is chosen so that three CTAs still fit an SM.
// Rows each thread keeps in flight (eight are never faster, and beyond 150 bins cost the third CTA: 200 bins of 2048 x 8192 33 us against 23).
constexpr int kHistAhead = 4;
constexpr int kHistStatic = 768;              // bytes of the kernel's fixed arrays
constexpr size_t kHistRoom = (228 * 1024 / 3 - 1024 - kHistStatic) / 256 * 256;     // dynamic shared memory of one of three CTAs on an SM (1 KB is set aside for each)
template <int R>
__global__ void __launch_bounds__(256, 3) histogram_kernel(const __half *__restrict__ X, int T, int C, long ldx,
                                                           int rows_per_split, int bins, const double *__restrict__ lo,
                                                           const double *__restrict__ hi, unsigned int *__restrict__ counts) {
    extern __shared__ __align__(16) unsigned int s_cnt[];   // [8][bins][8][R] | the threads' load rings: [kHistAhead + 1][256] x 16 bytes
    __shared__ float s_neg_lo[64], s_r[64];
    __shared__ __half s_lo[64], s_hi[64];
    static_assert(sizeof(s_neg_lo) + sizeof(s_r) + sizeof(s_lo) + sizeof(s_hi) == kHistStatic, "counted in kHistRoom");
    for (int i = threadIdx.x; i < 64 * R * bins; i += 256) s_cnt[i] = 0;
    grid_dependency_wait();
    grid_launch_dependents();
    // Exact bin: floor of the fp64 quotient q = (x - lo) * K / (hi - lo).  Almost every element gets there with one fp32
    // subtraction and one fused multiply-add (two elements per instruction), and no float <-> integer conversion (those run at a
    // quarter of the fp32 rate): with 2^S the largest power of two such that K * 2^S <= 2^22 and r = K * 2^S / (hi - lo) rounded once,
    //     t = fma(x - lo, r, 2^23 + 2)
    // lies in [2^23, 2^24), where floats are the integers, so the low 23 bits of t ARE n + 2 with n = round((x - lo) * r), and
    // |n - q * 2^S| <= 1: the subtraction (lo is exact in fp32) and r are each within 2^-24 relative, together at most
    // q * 2^S * 2^-23 <= 1/2, and the fma rounds once to an integer, at most 1/2.  So wherever n + 2 mod 2^S is 4 or more, bits S and
    // up of t are the exact bin.  The other elements (4 in 2^S: about one in ten thousand for a hundred bins, and always the
    // channel's minimum and maximum) take the fp64 division.  Elements are first clamped to the channel's range (two per
    // instruction), which bounds the counter's address whatever the input; a channel without a usable r (constant, or a range
    // that is not finite) is clamped to zero with r = 0, so n = 0 sends every element to the fp64 path.
    const int S = 22 - (32 - __clz(bins - 1));                                // bins >= 2
    if (threadIdx.x < 64 && blockIdx.x * 64 + threadIdx.x < C) {
        const int c = blockIdx.x * 64 + threadIdx.x;
        const double dl = lo[c], dh = hi[c], rng = __dsub_rn(dh, dl);
        float l = (float)dl, r = (float)(((double)bins / rng) * (double)(1 << S));
        __half cl = __float2half_rn(l), ch = __float2half_rn((float)dh);
        if (!(rng > 0.0 && rng < 1e6) || !(r <= 0x1p60f) || (double)__half2float(cl) != dl || (double)__half2float(ch) != dh) {
            l = r = 0.f;
            cl = ch = __ushort_as_half((unsigned short)0);
        }
        s_neg_lo[threadIdx.x] = -l;
        s_r[threadIdx.x] = r;
        s_lo[threadIdx.x] = cl;
        s_hi[threadIdx.x] = ch;
    }
    __syncthreads();
    const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
    const int cl = tx * 8;
    const int c0 = blockIdx.x * 64 + cl;
    const int r_begin = blockIdx.y * rows_per_split;
    const int r_end = min(T, r_begin + rows_per_split);
    if (c0 < C) {
        const unsigned int frac_mask = (1u << S) - 1u;
        uint64_t neg_lo[4], rf[4];
        __half2 lo_h[4], hi_h[4];
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) {
            neg_lo[k2] = f32x2(s_neg_lo[cl + 2 * k2], s_neg_lo[cl + 2 * k2 + 1]);
            rf[k2] = f32x2(s_r[cl + 2 * k2], s_r[cl + 2 * k2 + 1]);
            lo_h[k2] = __halves2half2(s_lo[cl + 2 * k2], s_lo[cl + 2 * k2 + 1]);
            hi_h[k2] = __halves2half2(s_hi[cl + 2 * k2], s_hi[cl + 2 * k2 + 1]);
        }
        const uint64_t magic = f32x2(8388610.f, 8388610.f);                  // 2^23 + 2
        // this thread's counter of bin -(2^23's bits >> S) for its first channel; the next channel's lies cnt_step bytes behind it
        const uint32_t cnt_0 = (uint32_t)__cvta_generic_to_shared(s_cnt + tx * R + (ty & (R - 1))) - (0x4B000000u >> S) * (uint32_t)(32 * R);
        const uint32_t cnt_step = (uint32_t)(bins * 32 * R);
        // One branch per row of eight elements, not one per element: the eight estimates are formed first, together with the
        // smallest distance-to-a-boundary code among them; only a row that holds an undecided element (about one row in a
        // thousand) goes back over its elements.
        auto count_row = [&](const uint4 &v) {
            const __half2 *h2 = reinterpret_cast<const __half2 *>(&v);
            unsigned int b[8], closest = 0xFFFFFFFFu;
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) {
                const float2 x = __half22float2(__hmin2(__hmax2(h2[k2], lo_h[k2]), hi_h[k2]));
                const uint64_t t = fma_f32x2(add_f32x2(f32x2(x.x, x.y), neg_lo[k2]), rf[k2], magic);
                const unsigned int t0 = (unsigned int)t, t1 = (unsigned int)(t >> 32);
                b[2 * k2] = t0 >> S;
                b[2 * k2 + 1] = t1 >> S;
                closest = min(closest, min(t0 & frac_mask, t1 & frac_mask));
            }
            if (closest < 4u) {
#pragma unroll
                for (int k2 = 0; k2 < 4; ++k2) {
                    const float2 x = __half22float2(__hmin2(__hmax2(h2[k2], lo_h[k2]), hi_h[k2]));
                    const uint64_t t = fma_f32x2(add_f32x2(f32x2(x.x, x.y), neg_lo[k2]), rf[k2], magic);
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        if (((unsigned int)(e ? t >> 32 : t) & frac_mask) < 4u)
                            b[2 * k2 + e] = (0x4B000000u >> S) + (unsigned int)histogram_exact_bin(__half2float(e ? __high2half(h2[k2]) : __low2half(h2[k2])),
                                                                                                  c0 + 2 * k2 + e, bins, lo, hi);
                }
            }
            uint32_t base = cnt_0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(base + (uint32_t)(32 * R) * b[k]) : "memory");
                base += cnt_step;
            }
        };
        // This thread's rows are r_begin + ty + 32 * i, i < n.  Loads and counting must overlap, and with 80 registers per thread
        // (three CTAs per SM) there is no room for a second set of rows in registers: every thread keeps kHistAhead of its own
        // 16-byte pieces in flight into a private slot ring in shared memory (asynchronous copies, one group per row; no
        // other thread touches the slots, so no barrier is needed).
        const int n = (r_end - r_begin - ty + 31) / 32;
        const __half *xcol = X + (long)(r_begin + ty) * ldx + c0;
        uint4 *ring = reinterpret_cast<uint4 *>(s_cnt + 64 * R * bins) + threadIdx.x;      // slot j of this thread: ring[256 * j]
        const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
        // (one slot more than rows in flight: the slot being refilled is the one read an iteration ago, whose values are used up)
        int wr = 0;
        auto fetch = [&](int i) {
            if (i < n)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ring_s + (uint32_t)(wr * 4096)),
                             "l"(xcol + (long)i * 32 * ldx)
                             : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");          // (an empty group past the end keeps the count in step)
            wr = wr == kHistAhead ? 0 : wr + 1;
        };
#pragma unroll
        for (int i = 0; i < kHistAhead; ++i) fetch(i);
        int rd = 0;
        for (int i = 0; i < n; ++i) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kHistAhead - 1) : "memory");
            const uint4 v = ring[256 * rd];
            rd = rd == kHistAhead ? 0 : rd + 1;
            fetch(i + kHistAhead);
            count_row(v);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int c = blockIdx.x * 64 + cl + k;
        for (int bin = ty; bin < bins; bin += 32) {
            const unsigned int *src = s_cnt + ((k * bins + bin) * 8 + tx) * R;
            unsigned int n = 0;
#pragma unroll
            for (int rep = 0; rep < R; ++rep) n += src[rep];
            if (c < C && n) atomicAdd(&counts[(long)c * bins + bin], n);
        }
    }
}

// Counter replicas for a bin count: one where a CTA has fewer than 512 rows, beyond as many as keep three CTAs on an SM (kHistRoom; with 109 or 110
// bins a limit of 75 KB let only two on: 2048 x 8192 of 110 bins 32 us, one replica 22).  Replicas are cleared and added up whatever the rows, and what they
// spare is small: 100 bins of N(0, 1), one against two, 342 rows 13.6 / 13.8 us, 683 rows 19.8 / 20.1 by itself but eight chunks of a calibration 259.6 / 258.9,
// 1366 rows 29.8 / 29.5, 2521 rows 47.4 / 45.5; 50 bins, one against four, 1366 rows 28.1 / 27.2, 2521 rows 45.8 / 42.4; all but a few elements in one or
// two bins: within 4 % either way.
// Token splits: whole waves of three CTAs per SM (the counting is bound by the shared-memory atomics, about 17 ns per token row of a CTA
// at that residency, so a partial wave is lost time; 2048 x 8192: 640 CTAs 30 us, 384 CTAs 20.5); a CTA's set-up and the addition of its counters to the
// global ones take as long as some 250 rows.
inline esp_status_t launch_histogram(const __half *X, int T, int C, long ldx, int bins, const double *lo, const double *hi, unsigned int *counts,
                                     int sm_count, cudaStream_t stream) {
    const size_t per_replica = sizeof(unsigned int) * 64 * (size_t)bins;
    const size_t ring = (size_t)(kHistAhead + 1) * 256 * 16;
    const int cols = ceil_div(C, 64), most = std::max(1, std::min(64, ceil_div(T, 32)));
    int splits = 1;
    long best = -1;
    for (int s = 1; s <= most; ++s) {
        const long cost = (long)ceil_div((long)cols * s, 3L * sm_count) * (ceil_div(T, s) + 250);
        if (best < 0 || cost < best) { best = cost; splits = s; }
    }
    const int rows = ceil_div(T, splits);
    const int R = rows < 512 ? 1 : per_replica * 4 + ring <= kHistRoom ? 4 : per_replica * 2 + ring <= kHistRoom ? 2 : 1;
    const size_t smem = per_replica * R + ring;
    auto kern = R == 4 ? histogram_kernel<4> : R == 2 ? histogram_kernel<2> : histogram_kernel<1>;
    ESP_CUDA_OK(ensure_dynamic_smem((const void *)kern, (int)smem));
    ESP_CUDA_OK(launch_overlapped(kern, dim3(cols, splits), 1, 256, smem, stream, X, T, C, ldx, rows, bins, lo, hi, counts));
    return ESP_OK;
}

// IR_c = -sum_k p_k ln p_k (Eq. 1, bins in index order, empty bins skipped) and s_c = IR_c + alpha*AM_c (Eq. 3).
// A CTA takes kEntropyChannels channels: all threads form the terms of its counts, then one thread per channel subtracts them in bin
// order, the order being part of the result.  (One thread per channel doing both, with strided reads, took 42 us whatever the size;
// this 11.)
struct EntropyOut {
    const double *norm, *sumsq;              // the norm is given, or the sum of squares it is the root of
    double *score;
    double *norm_out, *entropy_out, *score_out;      // copies for the caller, or NULL
};
constexpr int kEntropyChannels = 16;
__global__ void __launch_bounds__(256) entropy_score_kernel(int C, int T, int bins, const unsigned int *__restrict__ counts, double alpha,
                                                            int use_entropy, int use_norm, const double *__restrict__ score_override,
                                                            const EntropyOut out) {
    extern __shared__ double s_term[];       // [kEntropyChannels][bins | 1]
    const int c0 = blockIdx.x * kEntropyChannels, nc = min(kEntropyChannels, C - c0), ld = bins | 1;
    grid_dependency_wait();
    grid_launch_dependents();
    if (counts) {
        for (int i = threadIdx.x; i < nc * bins; i += 256) {
            const unsigned int n = counts[(long)c0 * bins + i];
            double term = 0.0;
            if (n) {                         // (few tokens leave most bins empty: dividing for those too, 36864 channels of 512 bins took 190 us, not 149)
                const double p = __ddiv_rn((double)n, (double)T);
                term = __dmul_rn(p, log(p));
            }
            s_term[(i / bins) * ld + i % bins] = term;
        }
    }
    __syncthreads();
    if ((int)threadIdx.x >= nc) return;
    const int c = c0 + threadIdx.x;
    double ir = 0.0;
    if (counts) {
#pragma unroll 4
        for (int k = 0; k < bins; ++k) ir = __dsub_rn(ir, s_term[threadIdx.x * ld + k]);
        if (out.entropy_out) out.entropy_out[c] = ir;
    }
    const bool have_norm = out.norm || out.sumsq;
    const double norm = out.sumsq ? sqrt(out.sumsq[c]) : have_norm ? out.norm[c] : 0.0;
    if (out.norm_out && have_norm) out.norm_out[c] = norm;
    double s = 0.0;
    if (score_override) {
        s = score_override[c];
    } else {
        if (use_entropy) s = __dadd_rn(s, ir);
        if (use_norm) s = __dadd_rn(s, __dmul_rn(alpha, norm));
    }
    out.score[c] = s;
    if (out.score_out) out.score_out[c] = s;
}
inline esp_status_t launch_entropy(int C, int T, int bins, const unsigned int *counts, const esp_prune_opts &o, const double *score_override,
                                   const EntropyOut &out, cudaStream_t stream) {
    const size_t smem = counts ? sizeof(double) * kEntropyChannels * (size_t)(bins | 1) : 0;
    ESP_CUDA_OK(ensure_dynamic_smem((const void *)entropy_score_kernel, (int)smem));
    ESP_CUDA_OK(launch_overlapped(entropy_score_kernel, dim3(ceil_div(C, kEntropyChannels)), 1, 256, smem, stream, C, T, bins, counts, o.alpha,
                                  o.use_entropy, o.use_norm, score_override, out));
    return ESP_OK;
}

// --------------------------------------------------------------------------------------------------
// K3: exact column sums of |W| (units of 2^-24) -> mean of the metric per channel (for the global shuffle), and / or the exact
// retained sums A_q of every group of 4 consecutive positions of an order (Eq. 5; theta NULL = the identity, read in the same
// 16-byte pieces).  The two share the pass over W.
// --------------------------------------------------------------------------------------------------
template <bool COLSUM, bool GROUPS>
__global__ void __launch_bounds__(256) colabs_kernel(const __half *__restrict__ W, int No, int C, long ldw, int rows_per_split,
                                                     const double *__restrict__ score, const int32_t *__restrict__ theta,
                                                     unsigned long long *__restrict__ colsum, unsigned long long *__restrict__ kept) {
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int c0 = (blockIdx.x * 32 + tx) * 8;
    const int r_begin = blockIdx.y * rows_per_split;
    const int r_end = min(No, r_begin + rows_per_split);
    long long acc[8] = {0, 0, 0, 0, 0, 0, 0, 0}, top[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (c0 < C) {
        int ch[8];
        double sc[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            ch[k] = GROUPS && theta ? theta[c0 + k] : c0 + k;
            sc[k] = GROUPS ? score[ch[k]] : 0.0;
        }
        auto load = [&](int r) -> uint4 {
            const uint16_t *row = reinterpret_cast<const uint16_t *>(W) + (long)r * ldw;
            if (!(GROUPS && theta)) return __ldg(reinterpret_cast<const uint4 *>(row + c0));
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = __ldg(row + ch[2 * k]) | ((uint32_t)__ldg(row + ch[2 * k + 1]) << 16);
            return make_uint4(w[0], w[1], w[2], w[3]);
        };
        auto add_row = [&](const uint4 &v) {
            const uint16_t *h = reinterpret_cast<const uint16_t *>(&v);
            long long f[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                f[k] = half_bits_abs_fixed(h[k]);
                if (COLSUM) acc[k] += f[k];
            }
            if constexpr (GROUPS) {
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    double xi[4];
                    int ahead[4] = {0, 0, 0, 0};
#pragma unroll
                    for (int k = 0; k < 4; ++k) xi[k] = __dmul_rn(half_bits_abs_to_double(h[4 * g + k]), sc[4 * g + k]);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (q != k) ahead[k] += (xi[q] > xi[k] || (xi[q] == xi[k] && q < k)) ? 1 : 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (ahead[k] < 2) top[4 * g + k] += f[4 * g + k];
                }
            }
        };
        // four rows in flight per thread
        int r = r_begin + ty;
        for (; r + 24 < r_end; r += 32) {
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = load(r + 8 * u);
#pragma unroll
            for (int u = 0; u < 4; ++u) add_row(v[u]);
        }
        for (; r < r_end; r += 8) add_row(load(r));
    }
    __shared__ long long s_acc[8][256 + 1];
    const int c = blockIdx.x * 256 + threadIdx.x;
    auto reduce = [&](const long long (&v)[8], unsigned long long *out) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 8; ++k) s_acc[ty][tx * 8 + k] = v[k];
        __syncthreads();
        if (c < C) {
            long long a = 0;
#pragma unroll
            for (int y = 0; y < 8; ++y) a += s_acc[y][threadIdx.x];
            atomicAdd(&out[c], (unsigned long long)a);         // integer: order-independent
        }
    };
    if constexpr (COLSUM) reduce(acc, colsum);
    if constexpr (GROUPS) reduce(top, kept);
}

__global__ void mean_metric_kernel(int C, int No, const unsigned long long *__restrict__ colsum,
                                   const double *__restrict__ score, double *__restrict__ mean) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    double a = __dmul_rn(__ll2double_rn((long long)colsum[c]), 0x1p-24);
    mean[c] = __ddiv_rn(__dmul_rn(score[c], a), (double)No);
}

// --------------------------------------------------------------------------------------------------
// K4: global naive shuffle.  rank(c) = number of channels ahead of c in a stable descending sort of the
// mean metric; the channel of rank r goes to group r mod G, slot r div G (neighbours in rank never share
// a group).
// --------------------------------------------------------------------------------------------------
// A CTA ranks 32 channels, each by eight threads over an eighth of the means (shared memory), so that the C^2 comparisons spread over C / 32
// CTAs: 57 -> 13 us for 4096 channels against a CTA of 256 channels with one thread each.
__global__ void __launch_bounds__(256) gns_rank_kernel(int C, const double *__restrict__ mean, int use_gns, int m_group,
                                                       int32_t *__restrict__ theta0, double *__restrict__ sorted_mean) {
    __shared__ double tile[2048];
    __shared__ int s_rank[32];
    const int c = blockIdx.x * 32 + (threadIdx.x & 31), part = threadIdx.x >> 5;
    if (!use_gns) {
        if (part == 0 && c < C) theta0[c] = c;
        return;
    }
    if (threadIdx.x < 32) s_rank[threadIdx.x] = 0;
    const double mine = (c < C) ? mean[c] : 0.0;
    int rank = 0;
    for (int base = 0; base < C; base += 2048) {
        __syncthreads();
        const int n = min(2048, C - base);
        for (int i = threadIdx.x; i < n; i += 256) tile[i] = mean[base + i];
        __syncthreads();
        // (the means of lower channels are ahead when equal, those of higher ones are not: two loops without an index compare)
        const int lo = part * 256, hi = min(n, lo + 256), split = min(max(c - base, lo), hi);
        int i = lo;
        for (; i < split; ++i) rank += tile[i] >= mine ? 1 : 0;
        for (; i < hi; ++i) rank += tile[i] > mine ? 1 : 0;
    }
    atomicAdd(&s_rank[threadIdx.x & 31], rank);
    __syncthreads();
    if (part == 0 && c < C) {
        const int G = C / m_group, r = s_rank[threadIdx.x];
        theta0[(r % G) * m_group + r / G] = c;
        sorted_mean[r] = mine;
    }
}

// Near-ties of the sort: neighbours in rank whose means differ by less than 1e-6 relative (the order of such a pair
// hangs on the last bits of the score).  counters[2] receives the count.
__global__ void __launch_bounds__(256) gns_near_tie_kernel(int C, const double *__restrict__ sorted_mean,
                                                           unsigned long long *__restrict__ counters) {
    const int r = blockIdx.x * 256 + threadIdx.x;
    unsigned int near = 0;
    if (r + 1 < C) {
        const double a = sorted_mean[r], b = sorted_mean[r + 1];
        near = __dsub_rn(a, b) < __dmul_rn(1e-6, fabs(a)) ? 1u : 0u;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) near += __shfl_xor_sync(0xFFFFFFFFu, near, off);
    if ((threadIdx.x & 31) == 0 && near) atomicAdd(&counters[2], (unsigned long long)near);
}

// --------------------------------------------------------------------------------------------------
// K5: local block shuffle (Algorithm 1 lines 3-14).
// --------------------------------------------------------------------------------------------------
#include "lbs_kernels.cuh"

// base[g] = V(g) from the retained sums of its four positions (theta NULL = the identity order).
__global__ void __launch_bounds__(256) group_values_kernel(const unsigned long long *__restrict__ kept, const double *__restrict__ score,
                                                           const int32_t *__restrict__ theta, int G, double *__restrict__ base) {
    const int g = blockIdx.x * 256 + threadIdx.x;
    if (g >= G) return;
    unsigned long long A[4];
    double s[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        A[k] = kept[4 * g + k];
        s[k] = score[theta ? theta[4 * g + k] : 4 * g + k];
    }
    base[g] = lbs_group_value(A, s);
}

// Eq. 5 objectives: the group values summed in group order, one order per CTA (base0, base1, base2 -> out[0..2]).  The additions are
// one serial chain by definition; the values are brought into shared memory first, so that the chain waits on nothing else (one
// thread reading them from L2 took 40 us for 1024 groups, this 8).
__global__ void __launch_bounds__(256) objective_kernel(int G, const double *__restrict__ base0, const double *__restrict__ base1,
                                                        const double *__restrict__ base2, double *__restrict__ out) {
    __shared__ double s[2048];
    const double *base = blockIdx.x == 0 ? base0 : blockIdx.x == 1 ? base1 : base2;
    double t = 0.0;
    for (int g0 = 0; g0 < G; g0 += 2048) {
        const int n = min(2048, G - g0);
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += 256) s[i] = base[g0 + i];
        __syncthreads();
        if (threadIdx.x == 0) {
#pragma unroll 16
            for (int i = 0; i < n; ++i) t = __dadd_rn(t, s[i]);
        }
    }
    if (threadIdx.x == 0) out[blockIdx.x] = t;
}

// --------------------------------------------------------------------------------------------------
// K6: 2-of-4 selection + compression.  One CTA per output row: the row is staged in shared memory, then
// each thread handles 8 permuted positions (2 groups): 4 kept values + 1 metadata byte.
// --------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) select_compress_kernel(const __half *__restrict__ W, int No, int C, long ldw,
                                                              const double *__restrict__ score,
                                                              const int32_t *__restrict__ theta,
                                                              __half *__restrict__ vals, uint8_t *__restrict__ meta,
                                                              unsigned long long *__restrict__ counters, int rows_per_cta) {
    // A CTA takes rows_per_cta consecutive output rows into shared memory; a thread then reads the permutation and the
    // scores of its eight positions ONCE and applies them to every one of those rows (with one row per CTA the two gathers
    // were six times the bytes of the row itself).
    extern __shared__ __align__(16) uint16_t s_rows[];                  // [rows_per_cta][C]
    const int j0 = blockIdx.x * rows_per_cta;
    const int nrows = min(rows_per_cta, No - j0);
    const int chunks_per_row = C / 8;
    for (int idx = threadIdx.x; idx < nrows * chunks_per_row; idx += 256) {
        const int r = idx / chunks_per_row, c = (idx - r * chunks_per_row) * 8;
        *reinterpret_cast<uint4 *>(s_rows + (size_t)r * C + c) =
            __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const uint16_t *>(W) + (long)(j0 + r) * ldw + c));
    }
    __syncthreads();
    unsigned int near = 0;
    for (int u = threadIdx.x; u < C / 8; u += 256) {
        int ch[8];
        double sc[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) { ch[k] = theta[u * 8 + k]; sc[k] = score[ch[k]]; }
        for (int r = 0; r < nrows; ++r) {
            const uint16_t *s_row = s_rows + (size_t)r * C;
            const long j = j0 + r;
            uint16_t out[4];
            unsigned int byte = 0;
#pragma unroll
            for (int gg = 0; gg < 2; ++gg) {
                uint16_t h[4];
                double xi[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    h[k] = s_row[ch[gg * 4 + k]];
                    xi[k] = __dmul_rn(half_bits_abs_to_double(h[k]), sc[gg * 4 + k]);
                }
                int kept[2], nk = 0;
                double second = 0.0, third = 0.0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    int ahead = 0;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q == k) continue;
                        ahead += (xi[q] > xi[k] || (xi[q] == xi[k] && q < k)) ? 1 : 0;
                    }
                    if (ahead < 2) { if (nk < 2) kept[nk] = k; ++nk; }
                    if (ahead == 1) second = xi[k];
                    if (ahead == 2) third = xi[k];
                }
                if (__dsub_rn(second, third) < __dmul_rn(1e-6, second)) ++near;
                out[gg * 2 + 0] = h[kept[0]];
                out[gg * 2 + 1] = h[kept[1]];
                byte |= (unsigned int)(kept[0] | (kept[1] << 2)) << (4 * gg);
            }
            uint2 packed;
            packed.x = (unsigned int)out[0] | ((unsigned int)out[1] << 16);
            packed.y = (unsigned int)out[2] | ((unsigned int)out[3] << 16);
            *reinterpret_cast<uint2 *>(reinterpret_cast<uint16_t *>(vals) + j * (C / 2) + u * 4) = packed;
            meta[j * (C / 8) + u] = (uint8_t)byte;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) near += __shfl_xor_sync(0xFFFFFFFFu, near, off);
    if ((threadIdx.x & 31) == 0 && near) atomicAdd(&counters[0], (unsigned long long)near);
}

// 4-of-8 selection + compression (the 4:8 pattern of the paper's Table 1; no tensor-core form exists for it, so the
// output is plain: 4 kept values per group in position order and one mask byte per group, bit p = position p kept).
// One CTA per output row, one thread per group of 8 permuted positions.
__global__ void __launch_bounds__(256) select_compress_48_kernel(const __half *__restrict__ W, int No, int C, long ldw,
                                                                 const double *__restrict__ score,
                                                                 const int32_t *__restrict__ theta,
                                                                 __half *__restrict__ vals, uint8_t *__restrict__ mask,
                                                                 unsigned long long *__restrict__ counters) {
    extern __shared__ uint16_t s_row[];
    const int j = blockIdx.x;
    const uint16_t *Wr = reinterpret_cast<const uint16_t *>(W) + (long)j * ldw;
    for (int c = threadIdx.x * 8; c < C; c += 256 * 8)
        *reinterpret_cast<uint4 *>(s_row + c) = __ldg(reinterpret_cast<const uint4 *>(Wr + c));
    __syncthreads();
    unsigned int near = 0;
    for (int u = threadIdx.x; u < C / 8; u += 256) {
        uint16_t h[8];
        double xi[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int c = theta[u * 8 + k];
            h[k] = s_row[c];
            xi[k] = __dmul_rn(half_bits_abs_to_double(h[k]), score[c]);
        }
        uint16_t out[4] = {0, 0, 0, 0};
        unsigned int byte = 0;
        int nk = 0;
        double fourth = 0.0, fifth = 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            int ahead = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (q == k) continue;
                ahead += (xi[q] > xi[k] || (xi[q] == xi[k] && q < k)) ? 1 : 0;
            }
            if (ahead < 4) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (e == nk) out[e] = h[k];
                ++nk;
                byte |= 1u << k;
            }
            if (ahead == 3) fourth = xi[k];
            if (ahead == 4) fifth = xi[k];
        }
        if (__dsub_rn(fourth, fifth) < __dmul_rn(1e-6, fourth)) ++near;
        uint2 packed;
        packed.x = (unsigned int)out[0] | ((unsigned int)out[1] << 16);
        packed.y = (unsigned int)out[2] | ((unsigned int)out[3] << 16);
        *reinterpret_cast<uint2 *>(reinterpret_cast<uint16_t *>(vals) + (long)j * (C / 2) + u * 4) = packed;
        mask[(long)j * (C / 8) + u] = (uint8_t)byte;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) near += __shfl_xor_sync(0xFFFFFFFFu, near, off);
    if ((threadIdx.x & 31) == 0 && near) atomicAdd(&counters[0], (unsigned long long)near);
}

// --------------------------------------------------------------------------------------------------
// K7: re-tile (vals, meta) into the layout the sparse MMA reads.
// Per (feature tile ft, channel tile kt) 18432 contiguous bytes:
//   [0, 16384)      128 rows x 128 bytes of kept values, 16-byte chunk q of row r stored at chunk q ^ (r & 7)
//                   (the 128-byte swizzle of a K-major shared-memory operand)
//   [16384, 18432)  128 lanes x 4 words; lane l, word c: low half = metadata of row (l&7) + 16*(l>>4), high half =
//                   that row + 8, for channels 32c + 16*((l>>3)&1) .. +16 of the tile (the order in which the
//                   tensor-memory copy lays 16 bytes per lane next to the accumulator lanes)
// --------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) pack_kernel(const __half *__restrict__ vals, const uint8_t *__restrict__ meta,
                                                   int No, int C, uint8_t *__restrict__ packed, int k_tiles) {
    const int kt = blockIdx.x, ft = blockIdx.y;
    uint8_t *tile = packed + ((long)ft * k_tiles + kt) * kTileBytes;
    const uint16_t *v16 = reinterpret_cast<const uint16_t *>(vals);
    const long half_c = C / 2, meta_c = C / 8;
    // values: 128 rows x 8 chunks
    for (int i = threadIdx.x; i < 128 * 8; i += 256) {
        const int r = i >> 3, q = i & 7;
        const long row = (long)ft * 128 + r;
        const long col = (long)kt * 64 + q * 8;      // in kept-value units
        uint4 v = make_uint4(0, 0, 0, 0);
        if (row < No && col + 8 <= half_c && (half_c & 7) == 0) {      // rows of vals are 16-byte aligned
            v = *reinterpret_cast<const uint4 *>(v16 + row * half_c + col);
        } else if (row < No && col < half_c) {
            uint16_t *p = reinterpret_cast<uint16_t *>(&v);
            for (int e = 0; e < 8; ++e) if (col + e < half_c) p[e] = v16[row * half_c + col + e];
        }
        *reinterpret_cast<uint4 *>(tile + r * 128 + ((q ^ (r & 7)) << 4)) = v;
    }
    // metadata: 128 lanes x 4 words
    for (int i = threadIdx.x; i < 128 * 4; i += 256) {
        const int l = i >> 2, c = i & 3;
        const int r_lo = (l & 7) + 16 * (l >> 4);
        const int khalf = (l >> 3) & 1;
        unsigned int word = 0;
#pragma unroll
        for (int hi = 0; hi < 2; ++hi) {
            const long row = (long)ft * 128 + r_lo + 8 * hi;
            const long mb = (long)kt * 16 + c * 4 + khalf * 2;   // metadata byte column
            unsigned int m16 = 0x4444u;                          // padding: legal nibbles, values are zero
            if (row < No) {
                unsigned int b0 = (mb < meta_c) ? meta[row * meta_c + mb] : 0x44u;
                unsigned int b1 = (mb + 1 < meta_c) ? meta[row * meta_c + mb + 1] : 0x44u;
                m16 = b0 | (b1 << 8);
            }
            word |= m16 << (16 * hi);
        }
        reinterpret_cast<unsigned int *>(tile + kTileValBytes)[l * 4 + c] = word;
    }
}

// K11: dense [No, C] in original channel order, zeros where pruned.
__global__ void __launch_bounds__(256) decompress_kernel(const __half *__restrict__ vals, const uint8_t *__restrict__ meta,
                                                         const int32_t *__restrict__ perm, int No, int C,
                                                         __half *__restrict__ out, long ldw) {
    const int j = blockIdx.x;
    const uint16_t *v16 = reinterpret_cast<const uint16_t *>(vals) + (long)j * (C / 2);
    uint16_t *o = reinterpret_cast<uint16_t *>(out) + (long)j * ldw;
    for (int g = threadIdx.x; g < C / 4; g += 256) {
        unsigned int byte = meta[(long)j * (C / 8) + (g >> 1)];
        unsigned int nib = (g & 1) ? (byte >> 4) : (byte & 0xF);
        int i0 = nib & 3, i1 = (nib >> 2) & 3;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            int c = perm ? perm[4 * g + k] : 4 * g + k;
            uint16_t v = 0;
            if (k == i0) v = v16[2 * g];
            if (k == i1) v = v16[2 * g + 1];
            o[c] = v;
        }
    }
}

}  // namespace

// ----------------------------------------------------------------------------------------------------
// Host side
// ----------------------------------------------------------------------------------------------------
static int pick_splits(int rows, int col_blocks, int sm_count) {
    // enough CTAs to fill the machine a few times over, each with a worthwhile slice of rows
    int want = ceil_div(4L * sm_count, col_blocks);
    int max_by_rows = ceil_div(rows, 64);
    int s = want < 1 ? 1 : want;
    if (s > max_by_rows) s = max_by_rows;
    if (s > 1024) s = 1024;
    return s < 1 ? 1 : s;
}

PruneWorkspace carve_prune_workspace(void *ws, int No, int C, int T, const esp_prune_opts &o) {
    PruneWorkspace w{};
    size_t off = 0;
    auto take = [&](size_t bytes) { void *p = ws ? (char *)ws + off : nullptr; off += align_up(bytes, 256); return p; };
    w.lo = (double *)take(sizeof(double) * C);
    w.hi = (double *)take(sizeof(double) * C);
    w.norm = (double *)take(sizeof(double) * C);
    w.score = (double *)take(sizeof(double) * C);
    w.mean = (double *)take(sizeof(double) * C);
    // cleared by one call: counters .. counts
    w.counters = (unsigned long long *)take(sizeof(unsigned long long) * 8);
    w.objective = (double *)take(sizeof(double) * 4);
    w.colsum = (unsigned long long *)take(sizeof(unsigned long long) * C);
    w.kept = (unsigned long long *)take(sizeof(unsigned long long) * C);
    if (o.use_lbs) {
        w.stride = (int)align_up((size_t)o.lbs_block, 8);
        w.live = (uint8_t *)take((size_t)ceil_div(C, o.lbs_block) * w.stride);
        w.handed = (int *)take(sizeof(int) * (size_t)ceil_div(C, o.lbs_block));
        w.handed_swaps = (int *)take(sizeof(int) * (size_t)ceil_div(C, o.lbs_block));
        w.widest = (int *)take(sizeof(int) * (size_t)ceil_div(C, o.lbs_block));
    }
    w.counts = (unsigned int *)take(sizeof(unsigned int) * (size_t)C * o.bins);
    w.cleared_bytes = w.counts ? (size_t)((char *)w.counts - (char *)w.counters) + sizeof(unsigned int) * (size_t)C * o.bins : 0;
    w.theta0 = (int32_t *)take(sizeof(int32_t) * C);
    w.sorted_mean = (double *)take(sizeof(double) * C);
    for (double *&base : w.base) base = (double *)take(sizeof(double) * (size_t)(C / 4 + 1));
    if (o.use_lbs) {
        const int nblocks = ceil_div(C, o.lbs_block);
        w.ldt = (long)align_up((size_t)No, 8);
        w.wt = (uint16_t *)take(sizeof(uint16_t) * (size_t)C * w.ldt);
        w.wb = (uint16_t *)take(sizeof(uint16_t) * ((size_t)nblocks * No + kBoundOver) * w.stride);
        w.irregular = (uint8_t *)take((size_t)nblocks * No);
        w.handed_pos = (int32_t *)take(sizeof(int32_t) * C);
        w.handed_list = (int *)take(sizeof(int) * (size_t)nblocks);
        w.table = (double *)take(sizeof(double) * (size_t)nblocks * kLbsGroups * 4 * kLbsMax);
    }
    w.total_bytes = off;
    return w;
}

esp_status_t launch_pack(const __half *vals, const uint8_t *meta, int No, int C, void *packed, cudaStream_t stream) {
    const int k_tiles = ceil_div(C, kTileK), f_tiles = ceil_div(No, kTileFeat);
    pack_kernel<<<dim3(k_tiles, f_tiles), 256, 0, stream>>>(vals, meta, No, C, (uint8_t *)packed, k_tiles);
    ESP_CUDA_OK(cudaGetLastError());
    return ESP_OK;
}

// ---- streaming calibration: state = sumsq | lo | hi | norm (f64[C] each) | counts u32[C][bins]
CalibState carve_calib_state(void *state, int C, int bins) {
    CalibState c{};
    size_t off = 0;
    auto take = [&](size_t bytes) { void *p = state ? (char *)state + off : nullptr; off += align_up(bytes, 256); return p; };
    c.sumsq = (double *)take(sizeof(double) * C);
    c.lo = (double *)take(sizeof(double) * C);
    c.hi = (double *)take(sizeof(double) * C);
    c.norm = (double *)take(sizeof(double) * C);
    c.counts = (unsigned int *)take(sizeof(unsigned int) * (size_t)C * bins);
    take(16 * 64 * (size_t)C);               // (unused: the size that callers rely on has room for 64 chunk partials per channel)
    c.total_bytes = off;
    return c;
}

esp_status_t launch_calib_reset(const CalibState &c, int C, int bins, cudaStream_t stream) {
    const long n = (long)C * bins;
    calib_reset_kernel<<<ceil_div(n, 256), 256, 0, stream>>>(C, bins, c.sumsq, c.lo, c.hi, c.counts);
    ESP_CUDA_OK(cudaGetLastError());
    return ESP_OK;
}

esp_status_t launch_calib_range(const CalibState &c, const __half *X, int T, int C, long ldx, cudaStream_t stream) {
    DeviceInfo di;
    esp_status_t st = device_info(&di);
    if (st != ESP_OK) return st;
    return launch_colstats(X, T, C, ldx, ColStatsOut{c.sumsq, nullptr, c.lo, c.hi}, di.sm_count, stream);
}

esp_status_t launch_calib_histogram(const CalibState &c, const __half *X, int T, int C, long ldx, int bins, cudaStream_t stream) {
    DeviceInfo di;
    esp_status_t st = device_info(&di);
    if (st != ESP_OK) return st;
    return launch_histogram(X, T, C, ldx, bins, c.lo, c.hi, c.counts, di.sm_count, stream);
}

esp_status_t launch_calib_finish(const CalibState &c, int C, int bins, long long T_total, const esp_prune_opts &o, double *chan_norm,
                                 double *chan_entropy, double *chan_score, cudaStream_t stream) {
    return launch_entropy(C, (int)T_total, bins, c.counts, o, nullptr, EntropyOut{nullptr, c.sumsq, chan_score, chan_norm, chan_entropy, nullptr}, stream);
}

esp_status_t launch_decompress(const __half *vals, const uint8_t *meta, const int32_t *perm, int No, int C,
                               __half *out, long ldw, cudaStream_t stream) {
    decompress_kernel<<<No, 256, 0, stream>>>(vals, meta, perm, No, C, out, ldw);
    ESP_CUDA_OK(cudaGetLastError());
    return ESP_OK;
}

esp_status_t launch_prune(const __half *W, int No, int C, long ldw, const __half *Xcal, int T, long ldx,
                          const esp_prune_opts &o, __half *vals, uint8_t *meta, int32_t *perm, void *packed,
                          double *chan_norm, double *chan_entropy, double *chan_score, esp_prune_stats *stats,
                          PruneWorkspace &w, cudaStream_t stream) {
    DeviceInfo di;
    esp_status_t st = device_info(&di);
    if (st != ESP_OK) return st;
    const int cthreads = 256;
    const int cblocks = ceil_div(C, cthreads);
    // (the counts, last of what is cleared, are only used by a statistics pass: 36864 channels of 512 bins without one, 1024 rows selected: 0.210 -> 0.199 ms)
    const bool stats_pass = Xcal && (o.score_override == nullptr || chan_norm || chan_entropy);
    ESP_CUDA_OK(cudaMemsetAsync(w.counters, 0, stats_pass ? w.cleared_bytes : (size_t)((char *)w.counts - (char *)w.counters), stream));

    if (stats_pass) {
        // K1
        st = launch_colstats(Xcal, T, C, ldx, ColStatsOut{nullptr, w.norm, w.lo, w.hi}, di.sm_count, stream);
        if (st != ESP_OK) return st;
        if (o.global_bin_range) global_range_kernel<<<1, 1024, 0, stream>>>(C, w.lo, w.hi);
        // K2
        st = launch_histogram(Xcal, T, C, ldx, o.bins, w.lo, w.hi, w.counts, di.sm_count, stream);
        if (st != ESP_OK) return st;
        st = launch_entropy(C, T, o.bins, w.counts, o, o.score_override, EntropyOut{w.norm, nullptr, w.score, chan_norm, chan_entropy, chan_score}, stream);
    } else {
        st = launch_entropy(C, T, o.bins, nullptr, o, o.score_override, EntropyOut{nullptr, nullptr, w.score, nullptr, nullptr, chan_score}, stream);
    }
    if (st != ESP_OK) return st;
    ESP_CUDA_OK(cudaGetLastError());

    // K3 + K4: the column sums for the global shuffle and, when objectives are asked for, the retained sums under the identity
    const int G = C / 4;
    const bool gns = o.use_gns && !o.perm_override;
    const int wsplits = pick_splits(No, ceil_div(C, 256), di.sm_count);
    const dim3 wgrid(ceil_div(C, 256), wsplits);
    const int wrows = ceil_div(No, wsplits);
    if (gns && stats) colabs_kernel<true, true><<<wgrid, 256, 0, stream>>>(W, No, C, ldw, wrows, w.score, nullptr, w.colsum, w.kept);
    else if (gns) colabs_kernel<true, false><<<wgrid, 256, 0, stream>>>(W, No, C, ldw, wrows, w.score, nullptr, w.colsum, w.kept);
    else if (stats) colabs_kernel<false, true><<<wgrid, 256, 0, stream>>>(W, No, C, ldw, wrows, w.score, nullptr, w.colsum, w.kept);
    if (gns) mean_metric_kernel<<<cblocks, cthreads, 0, stream>>>(C, No, w.colsum, w.score, w.mean);
    if (stats) group_values_kernel<<<ceil_div(G, 256), 256, 0, stream>>>(w.kept, w.score, nullptr, G, w.base[2]);
    // (a block of one group holds no pair of positions in different groups: nothing to swap.  4096 x 4096 in blocks of 4: 6.8 -> 0.21 ms)
    const bool lbs = o.use_lbs && o.lbs_block > 4;
    int32_t *theta0 = (lbs || stats) ? w.theta0 : perm;
    if (o.perm_override)
        ESP_CUDA_OK(cudaMemcpyAsync(theta0, o.perm_override, sizeof(int32_t) * C, cudaMemcpyDeviceToDevice, stream));
    else {
        gns_rank_kernel<<<ceil_div(C, 32), 256, 0, stream>>>(C, w.mean, o.use_gns, o.m_group, theta0, w.sorted_mean);
        if (o.use_gns && stats) gns_near_tie_kernel<<<ceil_div(C, 256), 256, 0, stream>>>(C, w.sorted_mean, w.counters);
    }
    ESP_CUDA_OK(cudaGetLastError());

    // K5
    if (lbs) {
        const int nblocks = ceil_div(C, o.lbs_block);
        const size_t row_bytes = sizeof(uint16_t) * (size_t)C;
        const bool few = No < 4;                                  // (see below)
        // rows per CTA: about 96 KB of shared memory (two CTAs per SM), and a grid of two CTAs per SM at least
        int gather_rows = (int)std::max<size_t>(1, std::min<size_t>(8, (96 * 1024) / row_bytes));
        gather_rows = std::max(1, std::min(gather_rows, No / (2 * std::max(1, di.sm_count))));
        ESP_CUDA_OK(ensure_dynamic_smem((const void *)lbs_gather_kernel, (int)(row_bytes * gather_rows)));
        lbs_gather_kernel<<<ceil_div(No, gather_rows), 256, row_bytes * gather_rows, stream>>>(W, No, C, ldw, w.score, w.theta0, o.lbs_block, w.stride, nblocks,
                                                                                               gather_rows, w.wb, w.handed, w.widest, w.live, few, w.handed_list, w.counters);
        lbs_transpose_kernel<<<dim3(ceil_div(C, 64), ceil_div(No, 64)), 256, 0, stream>>>(W, No, C, ldw, w.wt, w.ldt);
        // the swaps by bounds, but for one to three rows: their last question is about exchanges that move a kept product to another group, dozens of gains of rounding
        // noise, so every block would end in the exact kernels all the same (256..4096 channels, by bounds and to the end / exactly from the start: 1 row 0.64 / 0.60 ms,
        // 2 rows 1.28 / 1.04, 3 rows 1.39 / 1.18, 4 rows 1.43 / 1.43, 5 rows 1.39 / 1.55)
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        if (!few) {
            ESP_CUDA_OK(ensure_dynamic_smem((const void *)lbs_bound_table_kernel, (int)sizeof(LbsBoundTableSmem)));
            lbs_bound_table_kernel<<<dim3(ceil_div(o.lbs_block, 8), nblocks), kBoundTableThreads, sizeof(LbsBoundTableSmem), stream>>>(
                w.wb, w.wt, w.ldt, No, w.stride, w.score, w.theta0, C, o.lbs_block, w.handed, w.widest, w.live, w.table);
            ESP_CUDA_OK(ensure_dynamic_smem((const void *)lbs_bound_greedy_kernel, (int)lbs_bound_smem(kBoundMinCluster)));
            ESP_CUDA_OK(cudaFuncSetAttribute(lbs_bound_greedy_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            const int nc = lbs_cluster_size(lbs_bound_greedy_kernel, lbs_bound_config, kBoundMinCluster, {10.0, 0.022}, nblocks, No, di.device);
            lbs_bound_config(cfg, attr, nblocks, nc, stream);
            ESP_CUDA_OK(cudaLaunchKernelEx(&cfg, lbs_bound_greedy_kernel, (const uint16_t *)w.wb, (const uint16_t *)w.wt, w.ldt, No, w.stride,
                                           (const double *)w.score, (const int32_t *)w.theta0, C, o.lbs_block, o.lbs_max_swaps, w.table, perm, w.counters,
                                           (const int *)w.widest, (const uint8_t *)w.live, w.handed, w.handed_swaps, w.handed_pos, w.handed_list, nc));
        }
        // the exact kernels, on the blocks that were handed to them (without any, 8 us of empty launches, 4 with the first two set up under their
        // predecessors, which the smallest calls notice: 8 x 8 112 -> 108 us, by the exact kernels alone 107)
        auto mark = o.lbs_block <= 8 ? lbs_mark_kernel<8> : o.lbs_block <= 32 ? lbs_mark_kernel<32> : lbs_mark_kernel<kLbsMax>;
        ESP_CUDA_OK(launch_overlapped(mark, dim3(ceil_div(No, 64), nblocks), 1, 256, 0, stream, w.wb, No, w.stride, w.score, w.theta0, C, o.lbs_block, w.handed,
                                      w.irregular));
        ESP_CUDA_OK(ensure_dynamic_smem((const void *)lbs_table_kernel, (int)sizeof(LbsTableSmem)));
        ESP_CUDA_OK(launch_overlapped(lbs_table_kernel, dim3(o.lbs_block / 4, nblocks), 1, kTableThreads, sizeof(LbsTableSmem), stream, w.wb, w.wt, w.ldt, w.irregular, No,
                                      w.stride, w.score, w.theta0, C, o.lbs_block, w.handed, (few ? (int32_t *)nullptr : w.handed_pos), w.table, w.base[1]));
        ESP_CUDA_OK(ensure_dynamic_smem((const void *)lbs_greedy_kernel, (int)lbs_greedy_smem(kGreedyMinCluster)));
        ESP_CUDA_OK(cudaFuncSetAttribute(lbs_greedy_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        // How many blocks there is work in is not known here: none as a rule, one now and then, all of a weight made of ties.  Up to as many as large
        // clusters serve sooner they are launched in those, beyond that in the size for all blocks; the other launch's clusters leave at once (2 us).  One
        // block of the 16 of 4096 x 4096 (a weight that is not finite) 11.5 -> 8.6 ms for the whole call, 9.3 by the exact kernels alone; all sixteen handed
        // over before their first swap 3.72 ms as before (4.5 in large clusters).
        const LbsSwapCost cost{10.0, 0.055};
        const int sizes[2] = {lbs_cluster_size(lbs_greedy_kernel, lbs_greedy_config, kGreedyMinCluster, cost, few ? nblocks : 1, No, di.device),
                              lbs_cluster_size(lbs_greedy_kernel, lbs_greedy_config, kGreedyMinCluster, cost, nblocks, No, di.device)};
        const int caps[2] = {lbs_cluster_capacity(lbs_greedy_kernel, lbs_greedy_config, sizes[0], di.device),
                             lbs_cluster_capacity(lbs_greedy_kernel, lbs_greedy_config, sizes[1], di.device)};
        int most = nblocks;
        if (sizes[0] != sizes[1])                                 // (both then come from a capacity)
            for (most = 1; most < nblocks && cost.of(sizes[0], caps[0], most + 1, No) <= cost.of(sizes[1], caps[1], most + 1, No);) ++most;
        for (int all = 0; all < (most < nblocks ? 2 : 1); ++all) {
            lbs_greedy_config(cfg, attr, all ? nblocks : most, sizes[all], stream);
            ESP_CUDA_OK(cudaLaunchKernelEx(&cfg, lbs_greedy_kernel, (const uint16_t *)w.wb, (const uint16_t *)w.wt, w.ldt, (const uint8_t *)w.irregular, No,
                                           w.stride, (const double *)w.score, (const int32_t *)w.theta0, C, o.lbs_block, o.lbs_max_swaps, w.table,
                                           (const double *)w.base[1], perm, w.counters, (const int *)w.handed_list, (const int *)w.handed_swaps,
                                           (const int32_t *)(few ? nullptr : w.handed_pos), sizes[all], all ? most : 0, all ? nblocks : most));
        }
        if (stats) {
            // the objectives before and after (colabs_kernel, which gathers the permuted channels from W, took 47 us for each of the orders of a 4096 x 4096 weight);
            // a warp's lanes take eight rows each
            lbs_value_kernel<<<dim3(G, 2), 32 * std::min(kValueThreads / 32, ceil_div(No, 256)), 0, stream>>>(w.wt, w.ldt, No, w.score, w.theta0, perm, w.base[0],
                                                                                                              w.base[1]);
            objective_kernel<<<3, 256, 0, stream>>>(G, w.base[0], w.base[1], w.base[2], w.objective);
        }
    } else if (stats) {
        ESP_CUDA_OK(cudaMemsetAsync(w.kept, 0, sizeof(unsigned long long) * C, stream));
        colabs_kernel<false, true><<<wgrid, 256, 0, stream>>>(W, No, C, ldw, wrows, w.score, w.theta0, w.colsum, w.kept);
        group_values_kernel<<<ceil_div(G, 256), 256, 0, stream>>>(w.kept, w.score, w.theta0, G, w.base[0]);
        objective_kernel<<<3, 256, 0, stream>>>(G, w.base[0], w.base[0], w.base[2], w.objective);
        ESP_CUDA_OK(cudaMemcpyAsync(perm, w.theta0, sizeof(int32_t) * C, cudaMemcpyDeviceToDevice, stream));
    }
    ESP_CUDA_OK(cudaGetLastError());

    // K6 + K7
    const size_t row_smem = sizeof(uint16_t) * (size_t)C;
    // rows per CTA of the 2:4 kernel: as many as fit about 96 KB of shared memory (two CTAs per SM), eight at most
    // (and no more than leave the grid two CTAs per SM)
    int sel_rows = (int)std::max<size_t>(1, std::min<size_t>(8, (96 * 1024) / row_smem));
    sel_rows = std::max(1, std::min(sel_rows, No / (2 * std::max(1, di.sm_count))));
    ESP_CUDA_OK(ensure_dynamic_smem((const void *)select_compress_kernel, (int)(row_smem * sel_rows)));
    if (o.m_group == 8) {
        ESP_CUDA_OK(ensure_dynamic_smem((const void *)select_compress_48_kernel, (int)row_smem));
        select_compress_48_kernel<<<No, 256, row_smem, stream>>>(W, No, C, ldw, w.score, perm, vals, meta, w.counters);
    } else
        select_compress_kernel<<<ceil_div(No, sel_rows), 256, row_smem * sel_rows, stream>>>(W, No, C, ldw, w.score, perm, vals, meta,
                                                                                             w.counters, sel_rows);
    ESP_CUDA_OK(cudaGetLastError());
    if (packed) {
        st = launch_pack(vals, meta, No, C, packed, stream);
        if (st != ESP_OK) return st;
    }
    if (stats) {
        unsigned long long h_counters[8];
        double h_obj[4];
        ESP_CUDA_OK(cudaMemcpyAsync(h_counters, w.counters, sizeof(h_counters), cudaMemcpyDeviceToHost, stream));
        ESP_CUDA_OK(cudaMemcpyAsync(h_obj, w.objective, sizeof(h_obj), cudaMemcpyDeviceToHost, stream));
        ESP_CUDA_OK(cudaStreamSynchronize(stream));
        stats->near_tie_groups = (long long)h_counters[0];
        stats->near_tie_sort = (long long)h_counters[2];
        stats->near_tie_swaps = (long long)h_counters[3];
        stats->lbs_swaps_total = (long long)h_counters[1];
        stats->obj_identity = h_obj[2];
        stats->obj_after_gns = h_obj[0];
        stats->obj_after_lbs = h_obj[1];
    }
    return ESP_OK;
}

}  // namespace esp
