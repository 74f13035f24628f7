// Block shuffle by bounds: the swaps of lbs_kernels.cuh's exact kernels (Algorithm 1 lines 3-14, Eq. 5), found from fp32 sums with proven error
// bounds.  Included by lbs_kernels.cuh.
//
// What a swap has to know is which pair's exchange gains most, not by how much.  Let p1 >= p2 >= p3 >= p4 be a group's products |w| s in a row.  Without
// slot k the two largest of the three others are f1 >= f2 (f2 = p3 if k is among the first two, else p2), and with x in k's place the two largest sum to
// f1 + max(f2, x).  So what the group gains by it is
//     G(g, k <- x) = R - D_k,     R = sum over rows of max(0, |w_x| s_x - f2),     D_k = sum over rows of max(0, |w_k| s_k - p3),
// and a pair gains the sum of its two entries.  R costs ONE saturating fp32 fma and one addition per (row, candidate, slot): products are
// scaled to at most 1/2 in magnitude, so that the clamp at 0 is the fma's own, and the clamp at 1 never acts.  No ranks, no sort, no branch, no case for
// products that fp32 cannot tell apart: the sums are continuous where they cross.  Nothing here asks for scores of one sign.
//
// An entry G carries a bound E on its distance from the exact kernels' gain (their fp64 roundings included), and a pair's gain is
// kept as the interval [l, u] in directed rounding.  If the pair with the largest l leaves every other pair's u behind by more than the
// near-tie distance, it is the exact kernels' choice; if no u is positive, the block is done.  Otherwise (three swaps in a hundred on a LLaMA-7B-shaped
// projection, with two pairs in question) the pairs that may be the best or nearly tied with it are evaluated exactly, from integer sums.  More of them than
// kBoundCand (ties by the dozen: equal columns, scores that leave nothing to choose) and the block is handed to the exact kernels as it stands; so are, from the
// start, blocks with weights that are not finite or with scores beyond 2^+-300 or 2^200 apart (fp64 products of scaled scores are then no longer the scaled
// products).
//
// E, in units of 2^-24.  A product that stays is rounded once (bound_split), a candidate's takes the rounding of its score; the fma rounds once.  Rounding
// preserves order, so the computed p2 and p3 are within one unit of theirs.  A clamped term of R, d = x - f2 > 0, is off by at most
// |x| + |f2| + d <= 2 d + 2 |f2| (2 |f2| where only the computed value is positive), one of D_k by 2 d + 2 |p3|.  Together 2 R + 2 D + 4 S with S the sum over
// rows of max(|p2|, |p3|) = max(p2, -p3).  An addition rounds by at most one unit of the partial sum, so R takes one unit per addition on its way (add_r): up to
// kBoundFold in a register, one per fold in shared memory, four in the tree over the warps; D (add_d) one per row of a thread, five in a warp, one per chunk, five
// over the warps; both five over the CTAs.  bound_of takes one unit more of R and two of D than that, and 1/85 of the whole: there second-order terms find room,
// and the 16 bits of mantissa that an entry gives up (bound_pack), 2^-36 of |R - D| = 2^-12 units of it.  (bound_shift makes room for them once more: E is at
// least five units of the entry, 2^-9 of it 2^-31.)  The last term, rows * 2^-49, is for the exact kernels' roundings: a group's value is at most the number of
// rows (two products of 1/2 in each), five roundings of 2^-53 in each of the four values of a gain and three in adding them make less than 26 * 2^-53 rows a
// pair; two entries have 32.  What is left of it (2^-51 rows a pair) is more than the underflow of products down to 2^-200 in fp32, 2^-132 a row, adds.
//
// Two channels whose products are all zero (score zero: dead inputs; column zero: pruned before) exchange for nothing: exactly 0 on both sides, so such
// entries carry no bound; otherwise dozens of them would stay in question to the end.  Columns of zeros count as scores of zero, which changes no product.
//
// What bounds it: on long slices instruction issue -- a row costs a warp 48 fma, 48 additions, 8 conversions and some 30 others for both groups (256
// candidates, 6 slots), about 20 ns of an SM's time where the exact kernels take 55 --, on short ones the latency of a swap (search, three cluster barriers,
// two trips to L2: about 9 us).  Against the exact kernels alone: the whole of esp_metric_prune on 4096 x 4096 9.6 -> 4.2 ms, 13824 x 5120
// 28.9 -> 12.4, 512 x 512 2.7 -> 1.4.

constexpr int kBoundAhead = 4;         // rows a warp keeps in flight
constexpr int kBoundCand = 32;         // pairs a swap evaluates exactly at most
constexpr int kBoundThreads = 512, kBoundWarps = kBoundThreads / 32, kBoundChunk = 1024, kBoundMinCluster = 4, kBoundMaxCluster = 16;
constexpr int kBoundFold = 32;         // rows of a warp between two additions to the sums in shared memory
constexpr int kBoundCells = 6 * kLbsMax;

// A value and its error bound in one word: the low 16 bits of the fp64 mantissa give way to the bound's upper half (rounded up).
__device__ __forceinline__ double bound_pack(double v, float e) {
    return __longlong_as_double((__double_as_longlong(v) & ~0xFFFFLL) | (long long)((__float_as_uint(e) + 0xFFFFu) >> 16));
}
__device__ __forceinline__ double bound_value(double p) { return __longlong_as_double(__double_as_longlong(p) & ~0xFFFFLL); }
__device__ __forceinline__ double bound_error(double p) { return (double)__uint_as_float((uint32_t)__double_as_longlong(p) << 16); }
// The bound of an entry R - D: additions on the way of R and of D, S (above), output rows.
__device__ __forceinline__ float bound_of(float R, int add_r, float D, int add_d, float S, int No) {
    const float units = __fadd_ru(__fadd_ru(__fmul_ru((float)(add_r + 3), R), __fmul_ru((float)(add_d + 4), D)), __fmul_ru(4.f, S));
    return __fmaf_ru(0x1.03p-24f, units, (float)No * 0x1p-49f);
}
// [l, u] of the gain of exchanging the channels behind two table entries.
__device__ __forceinline__ float2 bound_gain(double there, double back) {
    const double g = bound_value(there) + bound_value(back), e = bound_error(there) + bound_error(back);
    return make_float2(__double2float_rd(g - e), __double2float_ru(g + e));
}
// An entry of a group whose value has moved by the gain `by`.
__device__ __forceinline__ double bound_shift(double entry, double by) {
    return bound_pack(bound_value(entry) - bound_value(by), __double2float_ru((bound_error(entry) + bound_error(by)) * (1.0 + 0x1p-9)));
}

__device__ __forceinline__ float relu_fma(float a, float b, float c) {       // min(1, max(0, a b + c))
    float d;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// A score as the sum of two floats, the first of 12 bits: its product with an fp16 number is exact.
__device__ __forceinline__ float2 bound_split(double s) {
    const float hi = __uint_as_float(__float_as_uint((float)s) & 0xFFFFF000u);
    return make_float2(hi, (float)(s - (double)hi));
}
// Per row of a group: for each slot the threshold f2 its candidates have to pass (negated) and the row's term of D; the row's term of S.
__device__ __forceinline__ void bound_row(const uint16_t (&h)[4], const float2 *s, float (&neg)[4], float (&D)[4], float &size) {
    float a[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {                                 // (rounded once)
        const float w = __half2float(__ushort_as_half(h[k]));
        a[k] = __fmaf_rn(w, s[k].y, __fmul_rn(w, s[k].x));
    }
    const float h0 = fmaxf(a[0], a[1]), l0 = fminf(a[0], a[1]), h1 = fmaxf(a[2], a[3]), l1 = fminf(a[2], a[3]);
    const float y = fminf(h0, h1), z = fmaxf(l0, l1), p3 = fminf(y, z), p2 = fmaxf(y, z);
    size = fmaxf(p2, -p3);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        neg[k] = a[k] >= p2 ? -p3 : -p2;
        D[k] = fmaxf(__fsub_rn(a[k], p3), 0.f);
    }
}
// Sums of eight values over a warp; lane l gets the total of value l / 4.
__device__ __forceinline__ float warp_sums_8(float (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = 4; n >= 1; n >>= 1) {
        const bool up = lane & (n * 4);
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float keep = up ? v[i + n] : v[i], give = up ? v[i] : v[i + n];
            v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, n * 4);
        }
    }
    float t = v[0];
    t += __shfl_xor_sync(0xFFFFFFFFu, t, 2);
    return t + __shfl_xor_sync(0xFFFFFFFFu, t, 1);
}

// One warp's rows of a chunk: NT thresholds per row, 8 candidates per lane.  (Scalar additions: a packed one takes the pipe for two clocks as well and wants its
// operands in register pairs; 163 clocks for 48 fma and 24 packed additions, 131 with 48 scalar ones.)
template <int NT>
struct BoundSums {
    float acc[NT][8];
    float s[8];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[t][e] = 0.f;
    }
    __device__ __forceinline__ void row(const float (&w)[8], const float (&neg)[NT]) {
#pragma unroll
        for (int e = 0; e < 8; ++e)
#pragma unroll
            for (int t = 0; t < NT; ++t) acc[t][e] += relu_fma(w[e], s[e], neg[t]);
    }
    // cell (t, half, lane, q) of `to` belongs to candidate lane * 8 + half * 4 + q
    __device__ __forceinline__ void fold(float4 *to, bool first) {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const float *a = acc[t] + 4 * half;
                float4 v = make_float4(a[0], a[1], a[2], a[3]);
                float4 *cell = to + (t * 2 + half) * 32 + lane;
                if (!first) {
                    const float4 o = *cell;
                    v = make_float4(v.x + o.x, v.y + o.y, v.z + o.z, v.w + o.w);
                }
                *cell = v;
            }
    }
};
__device__ __forceinline__ int bound_cell_candidate(int c) { return ((c >> 2) & 31) * 8 + ((c >> 7) & 1) * 4 + (c & 3); }

// The rows warp, warp + warps, ... of a block's copy, kBoundAhead of them on their way into registers.  Lanes beyond the block read its first channels (their
// candidates do not exist).  Rows are asked for without a look at the last one: the copy has room for kBoundOver rows behind it, whatever is in them is not used.
constexpr int kBoundOver = 2 * kBoundAhead * kBoundWarps;
struct BoundFeed {
    uint4 buf[kBoundAhead];
    const uint16_t *next;              // this lane's piece of the next row to ask for
    uint32_t step;                     // halfs from one of the warp's rows to the next
    __device__ __forceinline__ void begin(const uint16_t *first) {
#pragma unroll
        for (int u = 0; u < kBoundAhead; ++u) buf[u] = __ldg(reinterpret_cast<const uint4 *>(first + (size_t)u * step));
        next = first + (size_t)kBoundAhead * step;
    }
    // row(i, its weights) for every row i, ... < n in turn (all but the last call take a multiple of four)
    template <typename Row>
    __device__ __forceinline__ void each(int i, int n, Row row) {
        auto one = [&](int i, int u, bool more) {
            float w[8];
            const __half2 *hp = reinterpret_cast<const __half2 *>(&buf[u]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 f = __half22float2(hp[k]);
                w[2 * k] = f.x;
                w[2 * k + 1] = f.y;
            }
            if (more) {
                buf[u] = __ldg(reinterpret_cast<const uint4 *>(next));
                next += step;
            }
            row(i, w);
        };
        static_assert(kBoundAhead == 4, "rows in fours");
#pragma unroll 1
        for (; i + 4 <= n; i += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) one(i + u, u, true);
        }
        // (the last few through the first slot, a loop so as not to fetch code for each of them)
#pragma unroll 1
        for (; i < n; ++i) {
            one(i, 0, false);
            buf[0] = buf[1];
            buf[1] = buf[2];
        }
    }
};

// Scores of a block scaled by a power of two so that its products |w| s come close to 1/2 and not beyond (`widest`: the bits of its largest |w|), zero for
// channels without a live weight.  Then a barrier.
__device__ __forceinline__ void bound_load_scores(const double *__restrict__ score, const int32_t *__restrict__ theta0, int p0, int m, int widest,
                                                  const uint8_t *__restrict__ live, double *s64, float *s32, int *top) {
    if (threadIdx.x == 0) *top = -100000;
    __syncthreads();
    for (int x = threadIdx.x; x < m; x += blockDim.x) atomicMax(top, ilogb(score[theta0[p0 + x]]));
    __syncthreads();
    const int e = *top + 3 + (widest ? ilogbf(__half2float(__ushort_as_half((unsigned short)widest))) : 0);
    for (int x = threadIdx.x; x < kLbsMax; x += blockDim.x) {
        const double s = x < m && live[x] ? scalbn(score[theta0[p0 + x]], -e) : 0.0;
        s64[x] = s;
        s32[x] = (float)s;
    }
    __syncthreads();
}

// ---- The first table: every (group, slot, candidate) of a block.  One CTA per (block, two groups), all rows.
constexpr int kBoundTableThreads = 256, kBoundTableWarps = kBoundTableThreads / 32;
struct LbsBoundTableSmem {
    float4 part[kBoundTableWarps][8 * 64];
    float4 neg[2][kBoundTableThreads];
    float D[2][kBoundTableWarps][8];                              // [4] is S
    double total[2][8];
    double s64[kLbsMax];
    float s32[kLbsMax];
    int top;
};
__global__ void __launch_bounds__(kBoundTableThreads, 2) lbs_bound_table_kernel(const uint16_t *__restrict__ Wb, const uint16_t *__restrict__ Wt, long ldt,
                                                                                int No, int stride, const double *__restrict__ score,
                                                                                const int32_t *__restrict__ theta0, int C, int lbs_block,
                                                                                const int *__restrict__ handed, const int *__restrict__ widest,
                                                                                const uint8_t *__restrict__ live, double *__restrict__ table) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    LbsBoundTableSmem &S = *reinterpret_cast<LbsBoundTableSmem *>(s_dyn);
    const int b = blockIdx.y, p0 = b * lbs_block, m = min(lbs_block, C - p0), q0 = blockIdx.x * 8;
    if (q0 >= m || handed[b]) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, x0 = lane * 8;
    BoundFeed feed;
    feed.step = (uint32_t)(kBoundTableWarps * stride);
    bound_load_scores(score, theta0, p0, m, widest[b], live + (size_t)b * stride, S.s64, S.s32, &S.top);
    BoundSums<8> sums;
#pragma unroll
    for (int e = 0; e < 8; ++e) sums.s[e] = S.s32[x0 + e];
    const uint16_t *wt[8];
    float2 sg[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int p = min(q0 + k, m - 1);                         // (a second group beyond the block repeats its last channel)
        wt[k] = Wt + (long)theta0[p0 + p] * ldt;
        sg[k] = bound_split(S.s64[p]);
    }
    uint16_t h[8];
    auto load = [&](int r) {
#pragma unroll
        for (int k = 0; k < 8; ++k) h[k] = r < No ? __ldg(wt[k] + r) : (uint16_t)0;
    };
    load(tid);
#pragma unroll 1
    for (int r0 = 0; r0 < No; r0 += kBoundTableThreads) {
        const int nrows = min(kBoundTableThreads, No - r0);
        const int n = (nrows - warp + kBoundTableWarps - 1) / kBoundTableWarps;
        feed.begin(Wb + ((size_t)b * No + r0 + warp) * stride + (x0 < stride ? x0 : 0));
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const uint16_t hg[4] = {h[4 * g], h[4 * g + 1], h[4 * g + 2], h[4 * g + 3]};
            float neg[4], D[4], v[8] = {};
            bound_row(hg, sg + 4 * g, neg, D, v[4]);              // (a row beyond the last has zeros everywhere)
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = D[k];
            S.neg[g][tid] = make_float4(neg[0], neg[1], neg[2], neg[3]);
            const float t = warp_sums_8(v);
            if ((lane & 3) == 0) S.D[g][warp][lane >> 2] = r0 == 0 ? t : S.D[g][warp][lane >> 2] + t;
        }
        __syncthreads();
        load(r0 + kBoundTableThreads + tid);
        sums.clear();
        feed.each(0, n, [&](int i, const float (&w)[8]) {
            const int r = warp + kBoundTableWarps * i;
            const float4 a = S.neg[0][r], c = S.neg[1][r];
            const float neg[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
            sums.row(w, neg);
        });
        sums.fold(S.part[warp], r0 == 0);
        __syncthreads();
    }
    if (tid < 16) {
        double t = 0.0;
        for (int w = 0; w < kBoundTableWarps; ++w) t += (double)S.D[tid >> 3][w][tid & 7];
        S.total[tid >> 3][tid & 7] = t;
    }
    __syncthreads();
    const int chunks = (No + kBoundTableThreads - 1) / kBoundTableThreads, add_r = min(kBoundTableThreads, No) / kBoundTableWarps + 1 + chunks + 3, add_d = 5 + chunks;
    const float *part = reinterpret_cast<const float *>(S.part);
    for (int c = tid; c < 8 * kLbsMax; c += kBoundTableThreads) {
        const int t = c >> 8, x = bound_cell_candidate(c);
        if (x >= m || q0 + t >= m) continue;
        float v[kBoundTableWarps];
#pragma unroll
        for (int w = 0; w < kBoundTableWarps; ++w) v[w] = part[w * 8 * kLbsMax + c];
#pragma unroll
        for (int n = kBoundTableWarps / 2; n >= 1; n >>= 1)
#pragma unroll
            for (int w = 0; w < n; ++w) v[w] += v[w + n];
        const double D = S.total[t >> 2][t & 3];
        const bool idle = S.s64[x] == 0.0 && S.s64[q0 + t] == 0.0;
        table[((long)b * kLbsGroups * 4 + q0 + t) * kLbsMax + x] =
            idle ? 0.0 : bound_pack((double)v[0] - D, bound_of(v[0], add_r, __double2float_ru(D), add_d, __double2float_ru(S.total[t >> 2][4]), No));
    }
}

// ---- The swaps.  One cluster of CTAs per block of positions; the output rows are dealt to its CTAs, and so are the pairs, (i, j) to rank
// i mod cluster size.  Three cluster barriers per swap: after every CTA's best pair has been sent to all, when the sums of all CTAs are
// complete, and when the 6 x 256 new entries, each formed by one of the CTAs, are in all; the table in L2 is only for the columns that a swap looks up
// (entries of other groups, asked for while the sums are being added).
struct LbsBoundSmem {
    float4 part[kBoundWarps][6 * 64];                             // the warps' sums; the CTA's end up in the first warp's
    union {
        struct { float4 neg_a[kBoundChunk]; float2 neg_b[kBoundChunk]; };
        double fresh[6][kLbsMax];                                 // the new entries, written by the CTAs of the cluster (the thresholds are used up)
    };
    float4 best[kBoundWarps], won[kBoundMaxCluster];              // (the latter written by the CTAs of the cluster)
    float D[kBoundWarps][8];                                      // of the six live slots; S of the two groups
    float D_of[kBoundMaxCluster][8];                              // written by the CTAs of the cluster
    unsigned long long exact[kBoundCand * 4][4];                  // this CTA's rows' sums
    double value[kBoundCand * 4];
    int list[kBoundMaxCluster][kBoundCand], list_n[kBoundMaxCluster];       // written by the CTAs of the cluster
    int found;
    float2 grp_s[8], split[kLbsMax];
    int grp_channel[8];
    double s64[kLbsMax];
    float s32[kLbsMax];
    int pos2x[kLbsMax], chan[kLbsMax], top;
    uint8_t own_row[kLbsMax];                                     // place of position i among the rows of this CTA's pairs, 255 = another CTA's
    float2 gains[1];                                              // [l, u]; [local rows] of m - 1 - i pairs each
};
inline size_t lbs_bound_smem(int nc) {
    return sizeof(LbsBoundSmem) + sizeof(float2) * (size_t)lbs_gain_offset((kLbsMax + nc - 1) / nc, kLbsMax, 0, nc);
}

// The pair with the largest l, its u, and the largest u of all others.
struct BoundBest {
    float l, u, rest;
    int id;
    __device__ __forceinline__ void add(float l2, float u2, float rest2, int id2) {
        const bool up = l2 > l;
        rest = fmaxf(fmaxf(rest, rest2), up ? u : u2);
        l = up ? l2 : l;
        u = up ? u2 : u;
        id = up ? id2 : id;
    }
    __device__ __forceinline__ void warp() {
        auto key = [](float v) { const int i = __float_as_int(v); return i ^ ((i >> 31) & 0x7FFFFFFF); };
        auto value = [](int k) { return __int_as_float(k ^ ((k >> 31) & 0x7FFFFFFF)); };
        const int top = __reduce_max_sync(0xFFFFFFFFu, key(l));
        const int first = __ffs(__ballot_sync(0xFFFFFFFFu, key(l) == top)) - 1;
        rest = value(__reduce_max_sync(0xFFFFFFFFu, key((int)(threadIdx.x & 31) == first ? rest : fmaxf(rest, u))));
        l = value(top);
        u = __shfl_sync(0xFFFFFFFFu, u, first);
        id = __shfl_sync(0xFFFFFFFFu, id, first);
    }
};
// The pair behind place `at` of the gains of CTA `rank` (whole warp).
__device__ __forceinline__ int bound_pair_at(int at, int rank, int m, int nc) {
    const int rows = rank < m ? (m - rank + nc - 1) / nc : 0;
    int r = -1;
#pragma unroll
    for (int q = 0; q < (kLbsMax / kBoundMinCluster + 31) / 32; ++q) {
        const int row = q * 32 + (threadIdx.x & 31);
        r += __popc(__ballot_sync(0xFFFFFFFFu, row < rows && lbs_gain_offset(row, m, rank, nc) <= at));
    }
    const int i = rank + nc * r;
    return i * kLbsMax + at - lbs_gain_offset(r, m, rank, nc) + i + 1;
}

// Exact sums of one ordered group of four channels over the rows from 8 lo, eight in every step (a lane each; the warp's total is added to `to`).
// Slices begin at multiples of eight rows and the channel-major copy has zeros up to the next one.
__device__ __forceinline__ void bound_exact_sums(const uint16_t *__restrict__ Wt, long ldt, int lo, int step, int n, const int (&channel)[4],
                                                 const double (&s)[4], unsigned long long *to) {
    unsigned long long A[4] = {0, 0, 0, 0};
    float s32[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) s32[k] = (float)s[k];
    for (int r = 8 * (lo + (threadIdx.x & 31)); r < n; r += 8 * step) {
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = __ldg(reinterpret_cast<const uint4 *>(Wt + (long)channel[k] * ldt + r));
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            uint16_t h[4];
            float p[4];
            int ahead[4] = {0, 0, 0, 0};
            bool close = false;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t w = u < 2 ? v[k].x : u < 4 ? v[k].y : u < 6 ? v[k].z : v[k].w;
                h[k] = (uint16_t)(u & 1 ? w >> 16 : w);
                p[k] = __half2float(__ushort_as_half(h[k])) * s32[k];
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = a + 1; b < 4; ++b) {
                    const bool first = p[a] >= p[b];
                    const float most = fmaxf(fabsf(p[a]), fabsf(p[b]));
                    close = close || !(fabsf(p[a] - p[b]) > most * kLbsMargin && most >= 0x1p-110f);
                    ahead[a] += first ? 0 : 1;
                    ahead[b] += first ? 1 : 0;
                }
            if (close) {                                          // fp32 cannot tell (zeros among them)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    ahead[k] = 0;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (q != k)
                            ahead[k] += metric_ahead(__dmul_rn(half_bits_abs_to_double(h[q]), s[q]), q, __dmul_rn(half_bits_abs_to_double(h[k]), s[k]), k) ? 1 : 0;
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (ahead[k] < 2) A[k] += (unsigned long long)half_bits_abs_fixed(h[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) A[k] += __shfl_xor_sync(0xFFFFFFFFu, A[k], o);
        if ((threadIdx.x & 31) == k && A[k]) atomicAdd(to + k, A[k]);
    }
}

// value[o][g] = V(g) under order o (theta0, theta), for the objectives.  A CTA per (group, order), one launch that needs nothing cleared and adds nothing up
// in memory: sums per slot in memory, cleared before and turned into values behind, were four launches more, which a weight with two swaps to make
// noticed (512 x 512, two swaps: 165 -> 155 us a call; by the exact kernels, which have the values at hand, 158).
constexpr int kValueThreads = 256;
__global__ void __launch_bounds__(kValueThreads) lbs_value_kernel(const uint16_t *__restrict__ Wt, long ldt, int No, const double *__restrict__ score,
                                                                  const int32_t *__restrict__ theta0, const int32_t *__restrict__ theta,
                                                                  double *__restrict__ value0, double *__restrict__ value) {
    __shared__ unsigned long long s_sum[4];
    const int g = blockIdx.x;
    const int32_t *order = blockIdx.y ? theta : theta0;
    int channel[4];
    double s[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        channel[k] = order[4 * g + k];
        s[k] = score[channel[k]];
    }
    if (threadIdx.x < 4) s_sum[threadIdx.x] = 0;
    __syncthreads();
    bound_exact_sums(Wt, ldt, threadIdx.x & ~31, blockDim.x, No, channel, s, s_sum);
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned long long A[4] = {s_sum[0], s_sum[1], s_sum[2], s_sum[3]};
        (blockIdx.y ? value : value0)[g] = lbs_group_value(A, s);
    }
}

// The exact choice among the pairs whose u reaches `reach` (all threads of all CTAs, three barriers of the cluster): 1 with the pair and whether it is nearly tied, 0 if it
// gains nothing, -1 if there are too many.
__device__ __noinline__ int bound_settle(LbsBoundSmem &S, float reach, int my_rows, int m, int rank, int nc, const uint16_t *__restrict__ Wt,
                                         long ldt, int nrows, int &pair, bool &near_tie) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) S.found = 0;
    if (tid < kBoundCand * 16) (&S.exact[0][0])[tid] = 0;
    static_assert(kBoundCand * 16 <= kBoundThreads, "one sum per thread");
    __syncthreads();
    for (int r = warp; r < my_rows; r += kBoundWarps) {
        const int i = rank + nc * r;
        const float2 *gr = S.gains + lbs_gain_offset(r, m, rank, nc);
        for (int j = i + 1 + lane; j < m; j += 32) {
            const float2 g = gr[j - i - 1];
            if (g.y >= reach && g.y > 0.f) {                      // (who cannot gain is neither the best nor nearly tied with it)
                const int at = atomicAdd(&S.found, 1);
                if (at < kBoundCand)
                    for (int c = 0; c < nc; ++c) st_remote_s32(map_to_rank(smem_u32(&S.list[rank][at]), (uint32_t)c), i * kLbsMax + j);
            }
        }
    }
    __syncthreads();
    if (tid < nc) st_remote_s32(map_to_rank(smem_u32(&S.list_n[rank]), (uint32_t)tid), S.found);
    cluster_arrive();
    cluster_wait();
    int total = 0;
    for (int c = 0; c < nc; ++c) total += S.list_n[c];
    if (total > kBoundCand) return -1;
    auto candidate = [&](int i) {
        int c = 0;
        while (i >= S.list_n[c]) i -= S.list_n[c++];
        return S.list[c][i];
    };
    // four groups for each pair: both with the other's channel, both as they are
    auto group = [&](int task, int (&x)[4]) {
        const int ij = candidate(task >> 2), which = task & 1, at = which ? ij & 255 : ij >> 8, other = which ? ij >> 8 : ij & 255;
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = S.pos2x[(task & 2) == 0 && k == (at & 3) ? other : (at & ~3) + k];
    };
    const int parts = max(1, kBoundWarps / max(1, 4 * total));    // warps per group
    for (int w = warp; w < 4 * total * parts; w += kBoundWarps) {
        const int task = w / parts, part = w - task * parts;
        int x[4], channel[4];
        double s[4];
        group(task, x);
#pragma unroll
        for (int k = 0; k < 4; ++k) { channel[k] = S.chan[x[k]]; s[k] = S.s64[x[k]]; }
        bound_exact_sums(Wt, ldt, part * 32, parts * 32, nrows, channel, s, S.exact[task]);
    }
    cluster_arrive();
    cluster_wait();
    if (tid < 4 * total) {
        int x[4];
        double s[4];
        unsigned long long A[4] = {0, 0, 0, 0};
        group(tid, x);
        for (int c = 0; c < nc; ++c)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                unsigned long long v;
                asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(map_to_rank(smem_u32(&S.exact[tid][k]), (uint32_t)c)) : "memory");
                A[k] += v;
            }
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = S.s64[x[k]];
        S.value[tid] = lbs_group_value(A, s);
    }
    cluster_arrive();                                             // (the sums have been read)
    cluster_wait();
    double best = -INFINITY, second = -INFINITY;
    int id = 0x7FFFFFFF;
    if (lane < total) {
        const double *v = S.value + 4 * lane;
        best = __dsub_rn(__dadd_rn(v[0], v[1]), __dadd_rn(v[2], v[3]));
        id = candidate(lane);
    }
    static_assert(kBoundCand <= 32, "one pair per lane");
    lbs_warp_best(best, second, id);
    if (!(best > 0.0)) return 0;
    pair = id;
    near_tie = second > -INFINITY && __dsub_rn(best, second) < __dmul_rn(1e-6, fabs(best));
    return 1;
}

__global__ void __launch_bounds__(kBoundThreads, 1) lbs_bound_greedy_kernel(const uint16_t *__restrict__ Wb, const uint16_t *__restrict__ Wt, long ldt, int No,
                                                                            int stride, const double *__restrict__ score,
                                                                            const int32_t *__restrict__ theta0, int C, int lbs_block, int max_swaps,
                                                                            double *__restrict__ table, int32_t *__restrict__ theta, unsigned long long *__restrict__ counters,
                                                                            const int *__restrict__ widest, const uint8_t *__restrict__ live, int *__restrict__ handed, int *__restrict__ handed_swaps,
                                                                            int32_t *__restrict__ handed_pos, int *__restrict__ handed_list, int nc) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    LbsBoundSmem &S = *reinterpret_cast<LbsBoundSmem *>(s_dyn);
    const int b = blockIdx.x / nc, rank = (int)cluster_ctarank();
    const int p0 = b * lbs_block, m = min(lbs_block, C - p0);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, x0 = lane * 8;
    if (handed[b]) {                                              // (the same for the whole cluster: only the gathering kernel has written it)
        if (rank == 0) for (int x = tid; x < m; x += kBoundThreads) handed_pos[p0 + x] = x;
        return;
    }
    double *tb = table + (long)b * kLbsGroups * 4 * kLbsMax;
    for (int x = tid; x < m; x += kBoundThreads) {
        S.pos2x[x] = x;
        S.chan[x] = theta0[p0 + x];
        S.own_row[x] = x % nc == rank ? (uint8_t)(x / nc) : (uint8_t)255;
    }
    bound_load_scores(score, theta0, p0, m, widest[b], live + (size_t)b * stride, S.s64, S.s32, &S.top);           // (ends with a barrier: everything above is visible)
    for (int x = tid; x < m; x += kBoundThreads) S.split[x] = bound_split(S.s64[x]);          // (visible after the barrier below)
    const int per_cta = ((No + nc - 1) / nc + 7) & ~7, row0 = min(No, rank * per_cta), nrows_all = min(No, row0 + per_cta) - row0;
    const int add_r = min(kBoundFold, per_cta / kBoundWarps + 1) + per_cta / (kBoundWarps * kBoundFold) + 2 + 4 + 5;
    const int add_d = kBoundChunk / kBoundThreads + 5 + per_cta / kBoundChunk + 1 + 4 + 5;
    const uint16_t *wt_rows = Wt + row0;
    BoundSums<6> sums;
    BoundFeed feed;
    feed.step = (uint32_t)(kBoundWarps * stride);
    const uint16_t *wb_rows = Wb + ((size_t)b * No + row0 + warp) * stride + (x0 < stride ? x0 : 0);

    const int my_rows = rank < m ? (m - rank + nc - 1) / nc : 0, my_pairs = lbs_gain_offset(my_rows, m, rank, nc);
    for (int r = warp; r < my_rows; r += kBoundWarps) {
        const int i = rank + nc * r;
        float2 *gr = S.gains + lbs_gain_offset(r, m, rank, nc);
#pragma unroll 4
        for (int j = i + 1 + lane; j < m; j += 32) {
            const double there = __ldcg(&tb[i * kLbsMax + j]), back = __ldcg(&tb[j * kLbsMax + i]);
            gr[j - i - 1] = (i >> 2) == (j >> 2) ? make_float2(-INFINITY, -INFINITY) : bound_gain(there, back);
        }
    }
    // (a barrier of the cluster, not of the CTA: the first exchange below stores into the shared memory of the other CTAs, which have to be
    // running by then)
    cluster_arrive();
    cluster_wait();
    int swaps = 0, near_swaps = 0;
    bool hand_over = false;
    for (;;) {
        BoundBest best{-INFINITY, -INFINITY, -INFINITY, 0};
        if (max_swaps <= 0 || swaps < max_swaps) {
#pragma unroll 4
            for (int t = tid; t < my_pairs; t += kBoundThreads) {
                const float2 g = S.gains[t];
                best.add(g.x, g.y, -INFINITY, rank << 16 | t);
            }
        }
        best.warp();
        if (lane == 0) S.best[warp] = make_float4(best.l, best.u, best.rest, __int_as_float(best.id));
        __syncthreads();
        if (warp == 0) {
            const float4 v = S.best[lane & (kBoundWarps - 1)];
            best = lane < kBoundWarps ? BoundBest{v.x, v.y, v.z, __float_as_int(v.w)} : BoundBest{-INFINITY, -INFINITY, -INFINITY, 0};
            best.warp();
            if (lane < nc)                                        // this CTA's winner to every CTA of the cluster
                asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(map_to_rank(smem_u32(&S.won[rank]), (uint32_t)lane)), "f"(best.l),
                             "f"(best.u), "f"(best.rest), "f"(__int_as_float(best.id))
                             : "memory");
        }
        cluster_arrive();
        cluster_wait();
        {
            const float4 v = S.won[lane & (kBoundMaxCluster - 1)];
            best = lane < nc ? BoundBest{v.x, v.y, v.z, __float_as_int(v.w)} : BoundBest{-INFINITY, -INFINITY, -INFINITY, 0};
            best.warp();                                          // (every warp, the same result: no further exchange)
        }
        if (!(fmaxf(best.u, best.rest) > 0.f)) break;             // no pair can gain
        int pair;
        if (best.l > 0.f && best.rest < __fmul_rd(best.l, 1.f - 2e-6f)) pair = bound_pair_at(best.id & 0xFFFF, best.id >> 16, m, nc);
        else {                                                    // a near tie (1e-6) or closer than the bounds
            bool near_tie = false;
            const float reach = __fsub_rd(best.l, __fmul_ru(2e-6f, fmaxf(best.u, best.rest)));
            const int found = bound_settle(S, reach, my_rows, m, rank, nc, wt_rows, ldt, nrows_all, pair, near_tie);
            hand_over = found < 0;
            if (found <= 0) break;
            near_swaps += near_tie ? 1 : 0;                       // counted, not acted on
        }
        if (++swaps > kLbsSwapLimit) {
            if (tid == 0) atomicExch(&g_device_status, (int)ESP_ERR_TIMEOUT);
            break;
        }
        const int bi = pair >> 8, bj = pair & 255, ga = bi >> 2, gb = bj >> 2;
        const int xi = S.pos2x[bi], xj = S.pos2x[bj];             // (the channels that change places)
        const double by_a = __ldcg(&tb[bi * kLbsMax + xj]), by_b = __ldcg(&tb[bj * kLbsMax + xi]);      // what each group gains
        if (tid < 8) {
            const int p = (tid < 4 ? ga : gb) * 4 + (tid & 3), x = p == bi ? xj : p == bj ? xi : S.pos2x[p];
            S.grp_channel[tid] = S.chan[x];
            S.grp_s[tid] = S.split[x];
        }
        __syncthreads();
        if (tid == 0) { S.pos2x[bi] = xj; S.pos2x[bj] = xi; }
        // The six live slots: what a group is worth with a slot replaced depends on its OTHER three channels, so the swapped slots' rows of the table are only
        // shifted by what the group has gained (and offer the channel that left).
        const int skip_a = bi & 3, skip_b = bj & 3;
        bool first = true;
        int r0 = 0;
        do {
            const int nrows = min(kBoundChunk, nrows_all - r0);
            float total[8] = {};
            uint16_t h[kBoundChunk / kBoundThreads][8];
#pragma unroll
            for (int u = 0; u < kBoundChunk / kBoundThreads; ++u)
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int r = tid + u * kBoundThreads;
                    h[u][k] = r < nrows ? __ldg(wt_rows + (long)S.grp_channel[k] * ldt + r0 + r) : (uint16_t)0;
                }
#pragma unroll
            for (int u = 0; u < kBoundChunk / kBoundThreads; ++u) {
                if (warp * 32 + u * kBoundThreads >= nrows) break;
                float neg[6];
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    const uint16_t hg[4] = {h[u][4 * g], h[u][4 * g + 1], h[u][4 * g + 2], h[u][4 * g + 3]};
                    float t[4], D[4], size;
                    const int skip = g ? skip_b : skip_a;
                    bound_row(hg, S.grp_s + 4 * g, t, D, size);   // (a row beyond the slice has zeros everywhere)
                    total[6 + g] += size;
#pragma unroll
                    for (int l = 0; l < 3; ++l) {
                        neg[3 * g + l] = l >= skip ? t[l + 1] : t[l];
                        total[3 * g + l] += l >= skip ? D[l + 1] : D[l];
                    }
                }
                S.neg_a[tid + u * kBoundThreads] = make_float4(neg[0], neg[1], neg[2], neg[3]);
                S.neg_b[tid + u * kBoundThreads] = make_float2(neg[4], neg[5]);
            }
            if (warp * 32 < nrows) {
                const float t = warp_sums_8(total);
                if ((lane & 3) == 0) S.D[warp][lane >> 2] = first ? t : S.D[warp][lane >> 2] + t;
            } else if (first && lane < 8) S.D[warp][lane] = 0.f;
            __syncthreads();
            feed.begin(wb_rows + (size_t)r0 * stride);
#pragma unroll
            for (int e = 0; e < 8; ++e) sums.s[e] = S.s32[x0 + e];
            const int n = (nrows - warp + kBoundWarps - 1) / kBoundWarps;
            for (int i0 = 0; i0 < n || (first && i0 == 0); i0 += kBoundFold) {
                sums.clear();
                feed.each(i0, min(n, i0 + kBoundFold), [&](int i, const float (&w)[8]) {
                    const int r = warp + kBoundWarps * i;
                    const float4 a = S.neg_a[r];
                    const float2 c = S.neg_b[r];
                    const float n6[6] = {a.x, a.y, a.z, a.w, c.x, c.y};
                    sums.row(w, n6);
                });
                sums.fold(S.part[warp], first);
                first = false;
            }
            r0 += kBoundChunk;
            if (r0 < nrows_all) __syncthreads();
        } while (r0 < nrows_all);
        // the pairs of the eight positions of both groups: the entries that do not change are asked for now
        constexpr int kPer = 8 * kLbsMax / kBoundThreads;
        double there[kPer], back[kPer];
        int place[kPer];
        // entry (position p's slot, candidate x): NAN = among the new ones
        const bool skip_x = tid < 2 * kLbsMax && ((tid & 255) >> 5) % nc == rank && (tid & 255) < m;      // the swapped slots' entries that this CTA rewrites
        static_assert(kBoundThreads == 2 * kLbsMax, "an entry of the swapped slots per thread");
        double *skip_at = tb + (tid < kLbsMax ? bi : bj) * kLbsMax + (tid & 255);
        double skip_entry = skip_x ? __ldcg(skip_at) : 0.0;
        auto old_entry = [&](int p, int x) { return (p >> 2) != ga && (p >> 2) != gb || p == bi || p == bj ? __ldcg(&tb[p * kLbsMax + x]) : (double)NAN; };
        auto moved = [&](double e, int p, int x) {
            if ((p == bi || p == bj) && S.s64[x] == 0.0 && S.s64[p == bi ? xj : xi] == 0.0) return 0.0;
            return p == bi ? bound_shift(x == xi ? 0.0 : e, by_a) : p == bj ? bound_shift(x == xj ? 0.0 : e, by_b) : e;
        };
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int t = tid + u * kBoundThreads, which = t >> 8, p = (which < 4 ? ga : gb) * 4 + (which & 3), q = t & 255;
            const int i = min(p, q), j = max(p, q);
            place[u] = -1;
            const int row = S.own_row[i];
            if (j < m && (i >> 2) != (j >> 2) && row != 255) {
                place[u] = i * kLbsMax + j;
                there[u] = old_entry(i, S.pos2x[j]);
                back[u] = old_entry(j, S.pos2x[i]);
            }
        }
        __syncthreads();
        {
            float *part = reinterpret_cast<float *>(S.part);
#pragma unroll
            for (int u = 0; u < kBoundCells / kBoundThreads; ++u) {
                const int c = tid + u * kBoundThreads;
                float v[kBoundWarps];
#pragma unroll
                for (int w = 0; w < kBoundWarps; ++w) v[w] = part[w * kBoundCells + c];
#pragma unroll
                for (int n = kBoundWarps / 2; n >= 1; n >>= 1)
#pragma unroll
                    for (int w = 0; w < n; ++w) v[w] += v[w + n];
                part[c] = v[0];
            }
            if (warp == 0) {
                float t = 0.f;
#pragma unroll
                for (int w = 0; w < kBoundWarps / 4; ++w) t += S.D[(lane >> 3) * (kBoundWarps / 4) + w][lane & 7];
                t += __shfl_xor_sync(0xFFFFFFFFu, t, 8);
                t += __shfl_xor_sync(0xFFFFFFFFu, t, 16);
                for (int c = lane >> 3; c < nc; c += 4) st_remote_f32(map_to_rank(smem_u32(&S.D_of[rank][lane & 7]), (uint32_t)c), t);
            }
        }
        cluster_arrive();
        cluster_wait();                                           // the sums of every CTA are complete
        // this CTA forms `share` of the new entries and sends them to all (all of them formed by every CTA: 6150 clocks in a cluster of 6, 9980 in one of 16)
        const int share = ((kBoundCells + nc - 1) / nc + 31) & ~31;
        const int c = rank * share + tid;
        if (tid < share && c < kBoundCells) {
            const int t = c >> 8, x = bound_cell_candidate(c), g = t >= 3 ? 1 : 0, l = t - 3 * g, k = l + (l >= (g ? skip_b : skip_a) ? 1 : 0);
            const uint32_t cell = smem_u32(reinterpret_cast<const float *>(S.part) + c), to = smem_u32(&S.fresh[t][x]);
            float D = 0.f, T = 0.f, R = 0.f;
            auto tree = [](const float (&v)[8]) { return ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])); };
            for (int c0 = 0; c0 < nc; c0 += 8) {                  // (eight loads in flight)
                float v[8], d[8], u[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    v[r] = c0 + r < nc ? ld_dsmem_f32(cell, (uint32_t)(c0 + r)) : 0.f;
                    d[r] = c0 + r < nc ? S.D_of[c0 + r][t] : 0.f;
                    u[r] = c0 + r < nc ? S.D_of[c0 + r][6 + g] : 0.f;
                }
                D += tree(d);
                T += tree(u);
                R += tree(v);
            }
            const bool idle = S.s64[x] == 0.0 && S.grp_s[4 * g + k].x == 0.f;
            const double packed = idle ? 0.0 : bound_pack((double)R - (double)D, bound_of(R, add_r, D, add_d, T, No));
            for (int r = 0; r < nc; ++r) st_remote_f64(map_to_rank(to, (uint32_t)r), packed);
            if (x < m) tb[((g ? gb : ga) * 4 + k) * kLbsMax + x] = packed;
        }
        // (the swapped slots' entries are rewritten after the next barrier: they are used, and so have been read, before it)
        skip_entry = moved(skip_entry, tid < kLbsMax ? bi : bj, tid & 255);
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            if (place[u] < 0) continue;
            const int i = place[u] >> 8, j = place[u] & 255;
            there[u] = moved(there[u], i, S.pos2x[j]);
            back[u] = moved(back[u], j, S.pos2x[i]);
        }
        cluster_arrive();
        cluster_wait();                                           // the new entries are everywhere
        if (skip_x) *skip_at = skip_entry;
        auto fresh = [&](int p, int x) {
            const int g = (p >> 2) == ga ? 0 : 1, k = p & 3, skip = g ? skip_b : skip_a;
            return S.fresh[3 * g + k - (k > skip ? 1 : 0)][x];
        };
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            if (place[u] < 0) continue;
            const int i = place[u] >> 8, j = place[u] & 255;
            if (isnan(there[u])) there[u] = fresh(i, S.pos2x[j]);
            if (isnan(back[u])) back[u] = fresh(j, S.pos2x[i]);
            S.gains[lbs_gain_offset(S.own_row[i], m, rank, nc) + j - i - 1] = bound_gain(there[u], back[u]);
        }
        __syncthreads();
    }
    if (rank != 0) return;
    for (int x = tid; x < m; x += kBoundThreads) {
        theta[p0 + x] = S.chan[S.pos2x[x]];
        handed_pos[p0 + x] = S.pos2x[x];
    }
    if (tid == 0) {
        if (hand_over) { handed_swaps[b] = swaps; lbs_hand_over(b, handed, handed_list, counters); }
        if (swaps) atomicAdd(&counters[1], (unsigned long long)swaps);
        if (near_swaps) atomicAdd(&counters[3], (unsigned long long)near_swaps);
    }
}

inline void lbs_bound_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr, int nblocks, int nc, cudaStream_t stream) {
    lbs_greedy_config(cfg, attr, nblocks, nc, stream);
    cfg.blockDim = dim3(kBoundThreads);
    cfg.dynamicSmemBytes = lbs_bound_smem(nc);
}

// CTAs per block: the size that ends soonest, over waves of as many clusters as the device holds (asked once per kernel, size and device).
// A swap costs `fixed` us of barriers, search and exchange and `per_row` us per output row of a CTA's slice: about 10 and 0.055 by the exact kernel,
// 10 and 0.022 by bounds.
template <typename Kernel, typename Config>
inline int lbs_cluster_capacity(Kernel kernel, Config config, int nc, int device) {
    static std::mutex mu;
    static std::map<std::pair<const void *, int>, int> cache;
    std::lock_guard<std::mutex> lock(mu);
    const std::pair<const void *, int> key((const void *)kernel, device * 64 + nc);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    int cap = 0;
    config(cfg, attr, 1, nc, nullptr);
    if (cudaOccupancyMaxActiveClusters(&cap, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); cap = 0; }
    return cache[key] = cap;
}
struct LbsSwapCost {
    double fixed, per_row;
    double of(int nc, int capacity, int nblocks, int No) const {
        const double w = (double)nblocks / capacity, whole = std::ceil(w), waves = w <= 2.0 ? whole : w + (whole - w) * (2.0 / w);
        return waves * (fixed + per_row * (double)((No + nc - 1) / nc));
    }
};
template <typename Kernel, typename Config>
inline int lbs_cluster_size(Kernel kernel, Config config, int smallest, LbsSwapCost cost, int nblocks, int No, int device) {
    const int sizes[] = {16, 14, 12, 10, 9, 8, 7, 6, 5, 4, 3};
    int best = smallest;
    double best_cost = -1.0;
    for (int nc : sizes) {
        const int cap = nc < smallest ? 0 : lbs_cluster_capacity(kernel, config, nc, device);
        if (cap <= 0) continue;
        const double c = cost.of(nc, cap, nblocks, No);
        if (log_plans()) fprintf(stderr, "esparse block shuffle: blocks=%d rows=%d cluster=%d capacity=%d cost=%.1f\n", nblocks, No, nc, cap, c);
        if (best_cost < 0.0 || c < best_cost) { best_cost = c; best = nc; }
    }
    return best;
}
