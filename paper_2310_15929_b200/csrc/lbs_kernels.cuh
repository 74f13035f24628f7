// Local block shuffle (Algorithm 1 lines 3-14, Eq. 5): the exact kernels.  Included by prune_kernels.cu inside namespace esp { namespace { ... } }.
// lbs_bounds.cuh, included at the end, finds the same swaps from bounds; the kernels here take the blocks that it cannot decide, from the first swap or
// from where it stopped.
//
// Algorithm 1 needs, for every group g of a block, every slot k of g and every channel x of the block, the value
//   V(g, k <- x) = retained metric sum of g with slot k replaced by x
//                = ((s0*A0 + s1*A1) + s2*A2) + s3*A3,   A_q = sum of |w_q| over the rows in which slot q is among the 2 largest,
// where the A_q are exact integers of 2^-24 and "largest" is decided by the fp64 products |w| * s (ties: lower slot).  After every
// swap the values of the two touched groups change: 6 rows of 256 candidates, each a pass over all output rows of the weight.
// That pass is what the shuffle costs, and it is bound by instruction issue.  How the work per (row, candidate) is kept small:
//
//  * With the three fixed slots ranked f1, f2, f3 in a row, the candidate is kept exactly when it is ahead of f2; f1 is always
//    kept, f2 exactly when the candidate is not.  If the group's own four channels rank p1 > p2 > p3 > p4 in that row, f2 is p3 when
//    the replaced slot is p1 or p2, and p2 when it is p3 or p4: TWO comparisons per (row, candidate) serve all four slots.
//  * Rows are sorted by that rank order (24 classes, a counting sort in shared memory).  Inside a class the comparisons, the
//    two sums of kept |w_x| and the two sums of displaced |w_f2| have fixed meanings, so the loop has no per-row case analysis;
//    a warp adds its sums into per-slot totals when the class changes.
//  * A lane owns 8 candidates and a warp one row at a time: the row's record is uniform, a row of the block's gathered copy is
//    one 512-byte load, nothing is exchanged between lanes.
//  * fp32 products decide.  Each is within 2^-23 relative of its fp64 counterpart, so they order a row's channels as the fp64
//    products do unless two of them are closer than 2^-21.  Which rows hold such a pair is found once, in the blocks that come here (lbs_mark_kernel;
//    the products of a row's 256 channels never change, only their grouping does): those rows -- about one in a hundred where
//    the scores of a block differ -- and the rows with a magnitude of 0.5 or more are "irregular" and take fp64 products and
//    64-bit sums in a loop of their own.  Equal scores make nearly every row irregular, as do weights with sigma of 0.2 and more and, in
//    its block, a score that is not positive: little of the gain is left there.
//  * |w| < 0.5 becomes an integer of 2^-24 with one fp32 fma, so the sums are 32-bit adds.
//
// Measured, all blocks by these kernels, against one comparison and two fp64 additions per (row, candidate, slot) with a warp per candidate (about 29
// instructions each): table of a 4096 x 4096 weight 6.94 -> 0.92 ms, greedy kernel 67.7 -> 8.7 ms; 13824 x 5120: 29.1 -> 3.8 ms and 223 -> 24.4 ms; 512 x 512
// (two blocks): 15.6 -> 2.6 ms; to the end, 4096 x 4096 of irregular rows: 68.7 -> 57.0 ms with equal scores, 68.2 -> 51.8 at sigma 0.2.  (By bounds 4 ms,
// all of those.)

constexpr int kLbsMax = 256;       // widest local-shuffle block
constexpr int kLbsGroups = kLbsMax / 4;
constexpr int kLbsIrregular = 24;  // sort class of irregular rows, behind the 24 rank orders
constexpr uint16_t kWideBits = 0x3800;                     // |w| >= 0.5
constexpr float kLbsMargin = 0x1p-21f;

struct LbsRec {                    // one row of one group: the slots ranked second and third
    float p2, p3;                  // their products
    uint32_t u2, u3;               // their |w|: integers of 2^-24, in an irregular row fp16 bits
};
// A short slice's regular rows (lbs_thin): per live slot the product to beat, and what the candidate then displaces from each of the
// three other slots (one of them, zero from the rest).
constexpr int kThinRows = 192, kThinBatch = 16;
template <int NS>
struct __align__(16) LbsThinRec {
    float bound[NS];
    uint32_t u[NS][3];
};
template <int ROWS>
struct LbsRows {                   // the rows of a chunk as one group sees them, sorted by class
    union {
        LbsRec rec[ROWS];
        struct { LbsThinRec<4> thin[kThinRows + kThinBatch]; LbsRec thin_irregular[kThinRows]; };
    };
    uint16_t row[ROWS];
    uint16_t h1[ROWS];             // |w| bits of the slot ranked first
    uint8_t order[ROWS];           // rank order
    int cnt[32];
    int off[33];                   // first sorted place of a class
};
struct LbsGroup {                  // a group's four channels and their scores
    int channel[4];
    float s32[4];
    double s[4];
};
// Sums live in shared memory as 64-bit cells, low and high words apart: [cell][256 candidates], candidate x of lane x / 8 at
// (x & 7) * 32 + x / 8 (the lanes of a warp then add to consecutive words; the high words are only touched on a carry).
// Cells of a group with NS live slots (`skip` = the slot left out, or -1): NS sums of kept |w_x|, then for each slot the
// displaced sums of the three other slots.
template <int NS>
struct LbsCells {
    static constexpr int kCount = NS * 4, kWords = NS * 4 * kLbsMax;
    __device__ static int live(int k, int skip) { return NS == 4 ? k : k - (k > skip ? 1 : 0); }
    __device__ static int kept(int k, int skip) { return live(k, skip); }
    __device__ static int displaced(int k, int q, int skip) { return NS + live(k, skip) * 3 + (q < k ? q : q - 1); }
};
// Per group, beside the cells: M[q][p], the sum of |w_q| over the rows where slot q ranks third and slot p last (12 of them), then H[q],
// the sum over the rows where q is among the first two (4).
constexpr int kLbsGroupSums = 16;
__device__ __forceinline__ int lbs_third(int q, int p) { return q * 3 + (p < q ? p : p - 1); }

__device__ __forceinline__ bool metric_ahead(double xa, int sa, double xb, int sb) { return xa > xb || (xa == xb && sa < sb); }

// `n` = distance from the low to the high words.
__device__ __forceinline__ void lbs_add64(uint32_t *cell, int n, unsigned long long v) {
    const uint32_t lo = (uint32_t)v, hi = (uint32_t)(v >> 32);
    const uint32_t old = atomicAdd(cell, lo);
    const uint32_t up = hi + (old + lo < old ? 1u : 0u);
    if (up) atomicAdd(cell + n, up);
}
__device__ __forceinline__ unsigned long long lbs_cell(const uint32_t *cell, int n) { return ((unsigned long long)cell[n] << 32) | cell[0]; }

// Number of a rank order p1 > p2 > p3 > p4, and back.
__device__ __forceinline__ int lbs_order(int p1, int p2, int p3, int p4) { return p1 * 6 + (p2 - (p2 > p1 ? 1 : 0)) * 2 + (p3 > p4 ? 1 : 0); }
__device__ __forceinline__ void lbs_order_slots(int c, int &p1, int &p2, int &p3, int &p4) {
    p1 = c / 6;
    const int a = (c - 6 * p1) >> 1, r0 = p1 == 0 ? 1 : 0, r1 = p1 <= 1 ? 2 : 1, r2 = p1 <= 2 ? 3 : 2;
    p2 = a == 0 ? r0 : a == 1 ? r1 : r2;
    const int lo = a == 0 ? r1 : r0, hi = a == 2 ? r1 : r2;
    p3 = (c & 1) ? hi : lo;
    p4 = (c & 1) ? lo : hi;
}

template <typename T>
__device__ __forceinline__ T lbs_pick(const T (&v)[4], int i) { return i == 0 ? v[0] : i == 1 ? v[1] : i == 2 ? v[2] : v[3]; }

// Rank order and record of one row for one group.
__device__ __forceinline__ int lbs_classify(const uint16_t (&h)[4], const LbsGroup &grp, bool irregular, LbsRec &rec, uint16_t &h1) {
    float p[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) p[k] = __half2float(__ushort_as_half(h[k])) * grp.s32[k];
    int ahead[4] = {0, 0, 0, 0};                                  // slots ahead of this one
#pragma unroll
    for (int a = 0; a < 4; ++a) {
#pragma unroll
        for (int b = a + 1; b < 4; ++b) {
            bool first = p[a] >= p[b];                            // (equal only where both are zero: the lower slot)
            if (irregular)
                first = metric_ahead(__dmul_rn(half_bits_abs_to_double(h[a]), grp.s[a]), a, __dmul_rn(half_bits_abs_to_double(h[b]), grp.s[b]), b);
            ahead[a] += first ? 0 : 1;
            ahead[b] += first ? 1 : 0;
        }
    }
    int r1 = 0, r2 = 0, r3 = 0, r4 = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (ahead[k] == 0) r1 = k;
        if (ahead[k] == 1) r2 = k;
        if (ahead[k] == 2) r3 = k;
        if (ahead[k] == 3) r4 = k;
    }
    h1 = lbs_pick(h, r1);
    const uint16_t h2 = lbs_pick(h, r2), h3 = lbs_pick(h, r3);
    rec.p2 = lbs_pick(p, r2);
    rec.p3 = lbs_pick(p, r3);
    rec.u2 = irregular ? h2 : (uint32_t)half_bits_abs_fixed(h2);
    rec.u3 = irregular ? h3 : (uint32_t)half_bits_abs_fixed(h3);
    return min(lbs_order(r1, r2, r3, r4), 23);                    // (the bound only matters for NaN products, whose ranks are no order)
}

// Sorted records of NG groups over `nrows` <= ROWS rows.  Wt: the channel-major copy at the chunk's first row, so that the lanes of a
// warp read consecutive rows of a channel (from the gathered rows, 32 lanes would touch 32 lines per slot).  A thread keeps its
// records in registers from the count to the scatter.  `thin`: regular rows stay one class (see lbs_thin) and the group sums of all
// rows are added here; else those of the irregular ones.  The class counters are zero on entry and on return.
template <int NG, int ROWS, int THREADS, int NS>
__device__ __forceinline__ void lbs_prepare(const uint16_t *__restrict__ Wt, long ldt, const uint8_t *__restrict__ irregular, int nrows,
                                            const LbsGroup *grp, const int *skip, bool thin, LbsRows<ROWS> *rows, uint32_t *sums) {
    constexpr int kPer = NG * ROWS / THREADS;
    static_assert(kPer * THREADS == NG * ROWS && kPer <= 4, "rows per thread");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int total = NG * nrows;
    uint16_t h[kPer][4], h1[kPer];
    uint8_t irr[kPer];
    LbsRec rec[kPer];
    int where[kPer];                                              // order | class << 8 | place within the class << 16
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int i = tid + u * THREADS;
        if (i < total) {
            const int g = NG > 1 && i >= nrows ? 1 : 0, r = i - g * nrows;
#pragma unroll
            for (int k = 0; k < 4; ++k) h[u][k] = __ldg(Wt + (long)grp[g].channel[k] * ldt + r);
            irr[u] = __ldg(irregular + r);
        }
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int i = tid + u * THREADS;
        if (i < total) {
            const int g = NG > 1 && i >= nrows ? 1 : 0;
            const bool ir = irr[u] != 0;
            const int order = lbs_classify(h[u], grp[g], ir, rec[u], h1[u]), c = ir ? kLbsIrregular : thin ? 0 : order;
            where[u] = order | (c << 8) | (atomicAdd(&rows[g].cnt[c], 1) << 16);
            if (ir || thin) {
                int p1, p2, p3, p4;
                lbs_order_slots(order, p1, p2, p3, p4);
                uint32_t *sg = sums + g * 2 * kLbsGroupSums;
                lbs_add64(sg + 12 + p1, kLbsGroupSums, (unsigned long long)half_bits_abs_fixed(h1[u]));
                lbs_add64(sg + 12 + p2, kLbsGroupSums, ir ? (unsigned long long)half_bits_abs_fixed((uint16_t)rec[u].u2) : rec[u].u2);
                lbs_add64(sg + lbs_third(p3, p4), kLbsGroupSums, ir ? (unsigned long long)half_bits_abs_fixed((uint16_t)rec[u].u3) : rec[u].u3);
            }
        }
    }
    __syncthreads();
    if (warp < NG) {
        int v = rows[warp].cnt[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xFFFFFFFFu, v, o);
            if (lane >= o) v += t;
        }
        rows[warp].off[lane + 1] = v;
        if (lane == 0) rows[warp].off[0] = 0;
        rows[warp].cnt[lane] = 0;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int i = tid + u * THREADS;
        if (i < total) {
            const int g = NG > 1 && i >= nrows ? 1 : 0, at = rows[g].off[(where[u] >> 8) & 0xFF] + (where[u] >> 16);
            if (!thin) rows[g].rec[at] = rec[u];
            else if (irr[u]) rows[g].thin_irregular[at - rows[g].off[kLbsIrregular]] = rec[u];
            else {
                int p1, p2, p3, p4;
                lbs_order_slots(where[u] & 0xFF, p1, p2, p3, p4);
                LbsThinRec<NS> &t = reinterpret_cast<LbsThinRec<NS> *>(rows[g].thin)[at];
#pragma unroll
                for (int l = 0; l < NS; ++l) {
                    const int k = NS == 4 ? l : l + (l >= skip[g] ? 1 : 0);
                    const bool top = k == p1 || k == p2;
                    const int f2 = top ? p3 : p2;
                    t.bound[l] = top ? rec[u].p3 : rec[u].p2;
#pragma unroll
                    for (int o = 0; o < 3; ++o) t.u[l][o] = o + (o >= k ? 1 : 0) == f2 ? (top ? rec[u].u3 : rec[u].u2) : 0u;
                }
            }
            rows[g].row[at] = (uint16_t)(i - g * nrows);
            rows[g].h1[at] = h1[u];
            rows[g].order[at] = (uint8_t)where[u];
        }
    }
    if (thin && warp < NG) {                                      // the last batch is filled up
        const int at = rows[warp].off[kLbsIrregular] + lane;
        if (lane < kThinBatch) {
            LbsThinRec<NS> &t = reinterpret_cast<LbsThinRec<NS> *>(rows[warp].thin)[at];
#pragma unroll
            for (int l = 0; l < NS; ++l) {
                t.bound[l] = INFINITY;
                t.u[l][0] = t.u[l][1] = t.u[l][2] = 0u;
            }
        }
    }
    __syncthreads();
}

// What the regular rows [lo, hi) of one class (one warp, at most 128: 32-bit sums) add to their group's sums.
template <int ROWS>
__device__ __forceinline__ void lbs_group_sums(const LbsRows<ROWS> &R, int lo, int hi, int order, uint32_t *sums) {
    const int lane = threadIdx.x & 31;
    uint32_t v[3] = {0, 0, 0};
    for (int q = lo + lane; q < hi; q += 32) {
        v[0] += (uint32_t)half_bits_abs_fixed(R.h1[q]);
        v[1] += R.rec[q].u2;
        v[2] += R.rec[q].u3;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = __reduce_add_sync(0xFFFFFFFFu, v[i]);
    int p1, p2, p3, p4;
    lbs_order_slots(order, p1, p2, p3, p4);
    if (lane < 3) lbs_add64(sums + (lane == 0 ? 12 + p1 : lane == 1 ? 12 + p2 : lbs_third(p3, p4)), kLbsGroupSums, lane == 0 ? v[0] : lane == 1 ? v[1] : v[2]);
}

// 4 |w| + 2 is exact in fp32 for |w| < 0.5 and its bits are 2^30 + |w| 2^24, so sums of such bits are right in their low 30 bits (128
// values below 2^23) however many were added, and an addend costs one fma.
constexpr uint32_t kNarrowMask = 0x3FFFFFFFu, kNarrowBase = 0x40000000u;
constexpr int kNarrowRun = 128;
constexpr int kClassRows = 4;      // what the end of a class costs a warp, in rows
// Rows taken at once: equal chunks, and no more than leave every warp's run at 128 rows (see lbs_chunk).
__host__ __device__ constexpr int lbs_chunk_limit(int capacity) { return capacity - kClassRows * kLbsIrregular; }
__device__ __forceinline__ int lbs_chunk_rows(int n, int capacity) {
    const int chunks = max(1, (n + lbs_chunk_limit(capacity) - 1) / lbs_chunk_limit(capacity));
    return max(8, ((n + chunks - 1) / chunks + 7) & ~7);
}

// if (p > bound) { a += f; d += u; } as one comparison and two predicated additions (left to itself the compiler selects addends: four
// instructions instead of two).
__device__ __forceinline__ void lbs_count(uint32_t &a, uint32_t &d, uint32_t f, uint32_t u, float p, float bound) {
    asm("{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %4, %5;\n\t@p add.u32 %0, %0, %2;\n\t@p add.u32 %1, %1, %3;\n\t}"
        : "+r"(a), "+r"(d)
        : "r"(f), "r"(u), "f"(p), "f"(bound));
}
__device__ __forceinline__ int lbs_class_at(const int *off, int at) {        // the class whose rows include sorted place `at`
    return __popc(__ballot_sync(0xFFFFFFFFu, off[(threadIdx.x & 31) + 1] <= at));
}

// Regular rows [lo, hi) of the sorted order, at most 128 (one warp, 8 candidates per lane).  Rows arrive through a private ring in shared
// memory (asynchronous 16-byte copies, kRing - 1 rows ahead), which runs on across class boundaries; there the sums go to the cells.
// Classes c and c + 1 (c even) share p1 and p2: between them only the sums displaced from p3 have to leave the registers.
constexpr int kRing = 4;
template <int NS, int ROWS>
__device__ __forceinline__ void lbs_regular(const uint16_t *__restrict__ Wb, int stride, const LbsRows<ROWS> &R, int lo, int hi, int skip,
                                            const float *s32, uint4 *ring, uint32_t *cells, uint32_t *sums) {
    using Cells = LbsCells<NS>;
    const int lane = threadIdx.x & 31, x0 = lane * 8;
    const bool on = x0 < stride;
    uint64_t sx[4];
    uint32_t a2[8], d2[8], a3[8], d3[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) sx[i] = f32x2(s32[x0 + 2 * i], s32[x0 + 2 * i + 1]);
#pragma unroll
    for (int e = 0; e < 8; ++e) a2[e] = d2[e] = a3[e] = d3[e] = 0u;
    const uint64_t four = f32x2(4.f, 4.f), two = f32x2(2.f, 2.f);
    const uint32_t ring_s = smem_u32(ring + lane);                // slot j of this lane: ring[32 * j + lane]
    const uint16_t *wl = Wb + x0;
    auto fetch = [&](int q) {
        if (q < hi && on)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(ring_s + (uint32_t)(q % kRing) * 512u),
                         "l"(wl + (uint32_t)R.row[q] * (uint32_t)stride)
                         : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");      // (an empty group past the end keeps the count in step)
    };
    if (!on) {
#pragma unroll
        for (int j = 0; j < kRing; ++j) ring[32 * j + lane] = make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int j = 0; j < kRing - 1; ++j) fetch(lo + j);
    // adds sums of one kind to a slot's cells: eight returning additions in flight before their carries are looked at
    auto flush = [&](uint32_t *cell, const uint32_t (&v)[8], uint32_t mask) {
        uint32_t old[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) old[e] = atomicAdd(cell + lane + 32 * e, v[e] & mask);
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (old[e] + (v[e] & mask) < old[e]) atomicAdd(cell + lane + 32 * e + Cells::kWords, 1u);
    };
    int c = lbs_class_at(R.off, lo), run_lo = lo, run_hi = min(hi, R.off[c + 1]);
#pragma unroll 1
    for (int q = lo;;) {
#pragma unroll 1
        for (; q < run_hi; ++q) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");
            const uint4 v = ring[32 * (q % kRing) + lane];
            fetch(q + kRing - 1);                                 // (into the slot that was read one row ago)
            const LbsRec rec = R.rec[q];
            const __half2 *hp = reinterpret_cast<const __half2 *>(&v);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 w2 = __half22float2(hp[i]);
                const uint64_t w = f32x2(w2.x, w2.y), p = mul_f32x2(w, sx[i]), f = fma_f32x2(w, four, two);
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const int e = 2 * i + o;
                    const float pe = __uint_as_float((uint32_t)(o ? p >> 32 : p));
                    const uint32_t fe = (uint32_t)(o ? f >> 32 : f);
                    lbs_count(a2[e], d2[e], fe, rec.u2, pe, rec.p2);
                    lbs_count(a3[e], d3[e], fe, rec.u3, pe, rec.p3);
                }
            }
        }
        lbs_group_sums(R, run_lo, run_hi, c, sums);
        int p1, p2, p3, p4;
        lbs_order_slots(c, p1, p2, p3, p4);
        if (p1 != skip) flush(cells + Cells::displaced(p1, p3, skip) * kLbsMax, d3, 0xFFFFFFFFu);
        if (p2 != skip) flush(cells + Cells::displaced(p2, p3, skip) * kLbsMax, d3, 0xFFFFFFFFu);
#pragma unroll
        for (int e = 0; e < 8; ++e) d3[e] = 0u;
        const bool more = q < hi;
        const int next = more ? lbs_class_at(R.off, q) : 0;
        if (!more || (next >> 1) != (c >> 1)) {
            if (p1 != skip) flush(cells + Cells::kept(p1, skip) * kLbsMax, a3, kNarrowMask);
            if (p2 != skip) flush(cells + Cells::kept(p2, skip) * kLbsMax, a3, kNarrowMask);
            if (p3 != skip) { flush(cells + Cells::kept(p3, skip) * kLbsMax, a2, kNarrowMask); flush(cells + Cells::displaced(p3, p2, skip) * kLbsMax, d2, 0xFFFFFFFFu); }
            if (p4 != skip) { flush(cells + Cells::kept(p4, skip) * kLbsMax, a2, kNarrowMask); flush(cells + Cells::displaced(p4, p2, skip) * kLbsMax, d2, 0xFFFFFFFFu); }
            if (!more) break;
#pragma unroll
            for (int e = 0; e < 8; ++e) a2[e] = d2[e] = a3[e] = 0u;
        }
        c = next;
        run_lo = q;
        run_hi = min(hi, R.off[c + 1]);
    }
}

// ---- One candidate per lane (x; a group's candidates in eight warps), the per-slot totals in registers.
// The regular rows of a short slice, where a class would change every few rows and what that costs above would be most of the time:
// four predicated additions per live slot, whatever the row's rank order -- no branch (a jump by rank order took 550 clocks a row, most of
// them fetching instructions).
template <int NS, int ROWS>
__device__ __forceinline__ void lbs_thin(const uint16_t *__restrict__ Wb, int stride, const LbsRows<ROWS> &R, int nrows, int x, int skip,
                                         const float *s32, uint32_t *cells) {
    using Cells = LbsCells<NS>;
    const bool on = x < stride;
    const float sx = s32[x];
    const uint16_t *wl = Wb + x;
    const LbsThinRec<NS> *recs = reinterpret_cast<const LbsThinRec<NS> *>(R.thin);
    uint32_t kept[NS], displaced[NS][3];
#pragma unroll
    for (int l = 0; l < NS; ++l) kept[l] = displaced[l][0] = displaced[l][1] = displaced[l][2] = 0u;
    constexpr int kBatch = kThinBatch;                            // this many rows' weights at once, the next ones on their way meanwhile
    uint16_t cur[kBatch], next[kBatch];
    auto load = [&](int q) {
#pragma unroll
        for (int u = 0; u < kBatch; ++u) next[u] = on && q + u < nrows ? __ldg(wl + (uint32_t)R.row[q + u] * (uint32_t)stride) : (uint16_t)0;
    };
    load(0);
#pragma unroll 1
    for (int q0 = 0; q0 < nrows; q0 += kBatch) {
#pragma unroll
        for (int u = 0; u < kBatch; ++u) cur[u] = next[u];
        load(q0 + kBatch);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const LbsThinRec<NS> rec = recs[q0 + u];             // (beyond the last row: nothing is ahead of its bound)
            const float w = __half2float(__ushort_as_half(cur[u])), p = w * sx;
            const uint32_t f = __float_as_uint(fmaf(w, 4.f, 2.f)) - kNarrowBase;
#pragma unroll
            for (int l = 0; l < NS; ++l)
                asm("{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %8, %9;\n\t@p add.u32 %0, %0, %4;\n\t@p add.u32 %1, %1, %5;\n\t@p add.u32 %2, %2, %6;\n\t"
                    "@p add.u32 %3, %3, %7;\n\t}"
                    : "+r"(kept[l]), "+r"(displaced[l][0]), "+r"(displaced[l][1]), "+r"(displaced[l][2])
                    : "r"(f), "r"(rec.u[l][0]), "r"(rec.u[l][1]), "r"(rec.u[l][2]), "f"(p), "f"(rec.bound[l]));
        }
    }
    // (16 returning additions in flight before their carries are looked at)
    uint32_t *cell = cells + (x & 7) * 32 + (x >> 3);
    uint32_t old[NS][4];
#pragma unroll
    for (int l = 0; l < NS; ++l) {
        old[l][3] = atomicAdd(cell + l * kLbsMax, kept[l]);
#pragma unroll
        for (int o = 0; o < 3; ++o) old[l][o] = atomicAdd(cell + (NS + 3 * l + o) * kLbsMax, displaced[l][o]);
    }
#pragma unroll
    for (int l = 0; l < NS; ++l) {
        if (old[l][3] + kept[l] < kept[l]) atomicAdd(cell + l * kLbsMax + Cells::kWords, 1u);
#pragma unroll
        for (int o = 0; o < 3; ++o)
            if (old[l][o] + displaced[l][o] < displaced[l][o]) atomicAdd(cell + (NS + 3 * l + o) * kLbsMax + Cells::kWords, 1u);
    }
}

// Irregular rows [lo, hi): fp64 products, 64-bit sums, a branch on the row's rank order.
template <int P1, int P2, int P3, int P4>
__device__ __forceinline__ void lbs_add(unsigned long long (&kept)[4], unsigned long long (&displaced)[4][4], unsigned long long f, unsigned long long u2,
                                        unsigned long long u3, bool gt2, bool eq2, bool gt3, bool eq3) {
    if (gt3 || (eq3 && P1 < P3)) { kept[P1] += f; displaced[P1][P3] += u3; }
    if (gt3 || (eq3 && P2 < P3)) { kept[P2] += f; displaced[P2][P3] += u3; }
    if (gt2 || (eq2 && P3 < P2)) { kept[P3] += f; displaced[P3][P2] += u2; }
    if (gt2 || (eq2 && P4 < P2)) { kept[P4] += f; displaced[P4][P2] += u2; }
}
template <int NS, int ROWS>
__device__ __forceinline__ void lbs_exact(const uint16_t *__restrict__ Wb, int stride, const LbsRows<ROWS> &R, const LbsRec *recs, int lo, int hi, int x,
                                          const LbsGroup &grp, int skip, const double *s64, uint32_t *cells) {
    using Cells = LbsCells<NS>;
    const bool on = x < stride;
    const double sx = s64[x];
    const uint16_t *wl = Wb + x;
    unsigned long long kept[4] = {0, 0, 0, 0}, displaced[4][4] = {};
    auto load = [&](int q) -> uint16_t { return on && q < hi ? __ldg(wl + (uint32_t)R.row[q] * (uint32_t)stride) : (uint16_t)0; };
    uint16_t n0 = load(lo), n1 = load(lo + 1), n2 = load(lo + 2);  // the next rows' weights on their way
#pragma unroll 1
    for (int q = lo; q < hi; ++q) {
        const uint16_t hx = n0;
        n0 = n1;
        n1 = n2;
        n2 = load(q + 3);
        const int order = R.order[q];
        const LbsRec rec = recs[q - lo];
        int p1, p2, p3, p4;
        lbs_order_slots(order, p1, p2, p3, p4);
        const double xx = __dmul_rn(half_bits_abs_to_double(hx), sx);
        const double x2 = __dmul_rn(half_bits_abs_to_double((uint16_t)rec.u2), grp.s[p2]), x3 = __dmul_rn(half_bits_abs_to_double((uint16_t)rec.u3), grp.s[p3]);
        const bool gt2 = xx > x2, eq2 = xx == x2, gt3 = xx > x3, eq3 = xx == x3;
        const unsigned long long f = (unsigned long long)half_bits_abs_fixed(hx), u2 = (unsigned long long)half_bits_abs_fixed((uint16_t)rec.u2),
                                 u3 = (unsigned long long)half_bits_abs_fixed((uint16_t)rec.u3);
#define ESP_ORDER(N, P1, P2, P3, P4) case N: lbs_add<P1, P2, P3, P4>(kept, displaced, f, u2, u3, gt2, eq2, gt3, eq3); break;
        switch (order) {
            ESP_ORDER(0, 0, 1, 2, 3) ESP_ORDER(1, 0, 1, 3, 2) ESP_ORDER(2, 0, 2, 1, 3) ESP_ORDER(3, 0, 2, 3, 1) ESP_ORDER(4, 0, 3, 1, 2) ESP_ORDER(5, 0, 3, 2, 1)
            ESP_ORDER(6, 1, 0, 2, 3) ESP_ORDER(7, 1, 0, 3, 2) ESP_ORDER(8, 1, 2, 0, 3) ESP_ORDER(9, 1, 2, 3, 0) ESP_ORDER(10, 1, 3, 0, 2) ESP_ORDER(11, 1, 3, 2, 0)
            ESP_ORDER(12, 2, 0, 1, 3) ESP_ORDER(13, 2, 0, 3, 1) ESP_ORDER(14, 2, 1, 0, 3) ESP_ORDER(15, 2, 1, 3, 0) ESP_ORDER(16, 2, 3, 0, 1) ESP_ORDER(17, 2, 3, 1, 0)
            ESP_ORDER(18, 3, 0, 1, 2) ESP_ORDER(19, 3, 0, 2, 1) ESP_ORDER(20, 3, 1, 0, 2) ESP_ORDER(21, 3, 1, 2, 0) ESP_ORDER(22, 3, 2, 0, 1) ESP_ORDER(23, 3, 2, 1, 0)
            default: break;
        }
#undef ESP_ORDER
    }
    const int at = (x & 7) * 32 + (x >> 3);
    uint32_t old[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (k == skip) continue;
#pragma unroll
        for (int o = 0; o < 4; ++o)
            old[k][o] = atomicAdd(cells + (o == k ? Cells::kept(k, skip) : Cells::displaced(k, o, skip)) * kLbsMax + at, (uint32_t)(o == k ? kept[k] : displaced[k][o]));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (k == skip) continue;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const unsigned long long v = o == k ? kept[k] : displaced[k][o];
            const uint32_t up = (uint32_t)(v >> 32) + (old[k][o] + (uint32_t)v < (uint32_t)v ? 1u : 0u);
            if (up) atomicAdd(cells + (o == k ? Cells::kept(k, skip) : Cells::displaced(k, o, skip)) * kLbsMax + Cells::kWords + at, up);
        }
    }
}

// One chunk of rows, NG groups, into the cells and sums.
template <int NG, int ROWS, int THREADS, int NS>
__device__ __forceinline__ void lbs_chunk(const uint16_t *__restrict__ Wb, int stride, const uint16_t *__restrict__ Wt, long ldt,
                                          const uint8_t *__restrict__ irregular, int nrows, const LbsGroup *grp, const int *skip, LbsRows<ROWS> *rows,
                                          const float *s32, const double *s64, uint4 *ring, uint32_t *cells, uint32_t *sums) {
    constexpr int kWarps = THREADS / 32;
    static_assert(kWarps == 8 * NG, "a group's candidates in eight warps");
    static_assert(NG * (lbs_chunk_limit(ROWS) + kClassRows * kLbsIrregular) <= kNarrowRun * kWarps && kThinRows * (1ll << 23) < (1ll << 32), "32-bit sums");
    static_assert(sizeof(LbsThinRec<4>) * (kThinRows + kThinBatch) + sizeof(LbsRec) * kThinRows <= sizeof(LbsRec) * ROWS, "records of a short slice");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool thin = nrows <= kThinRows;
    lbs_prepare<NG, ROWS, THREADS, NS>(Wt, ldt, irregular, nrows, grp, skip, thin, rows, sums);
    const int mine = warp >> 3, x = lane * 8 + (warp & 7);        // group and candidate of this lane in the loops over single rows
    uint32_t *cells_mine = cells + mine * 2 * LbsCells<NS>::kWords;
    const LbsRows<ROWS> &R = rows[mine];
    const int regular = R.off[kLbsIrregular];
    // (half of the warps take the irregular rows first: that loop waits on memory and branches, the other fills the issue slots)
#pragma unroll 1
    for (int turn = 0; turn < 2; ++turn) {
        if ((turn ^ warp) & 1) {
            if (regular < nrows)
                lbs_exact<NS>(Wb, stride, R, thin ? R.thin_irregular : R.rec + regular, regular, nrows, x, grp[mine], skip[mine], s64, cells_mine);
        } else if (thin) {
            lbs_thin<NS>(Wb, stride, R, regular, x, skip[mine], s32, cells_mine);
        } else {
            // every warp a run of the groups' sorted regular rows, all candidates: equal shares of rows + kClassRows for every class that
            // has rows (a class ends with its sums going to the cells).  Equal numbers of rows leave the warps whose run crosses the
            // small classes far behind: a quarter of a swap was spent waiting for them (4096 x 4096 10.7 -> 10.1 ms, 3584 x 1224 5.63 -> 5.01 ms).
            int regular_rows[NG], at[NG + 1];                     // (cost before each group)
            uint32_t classes[NG];
            at[0] = 0;
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                regular_rows[g] = rows[g].off[kLbsIrregular];
                classes[g] = __ballot_sync(0xFFFFFFFFu, lane < kLbsIrregular && rows[g].off[lane + 1] > rows[g].off[lane]);
                at[g + 1] = at[g] + regular_rows[g] + kClassRows * __popc(classes[g]);
            }
#pragma unroll 1
            for (int g = 0; g < NG; ++g) {
                const int start = rows[g].off[lane] + kClassRows * __popc(classes[g] & ((1u << lane) - 1u));     // cost before class `lane`
                auto place = [&](int cost) {                      // the sorted place that this much cost reaches
                    cost = max(0, min(at[NG], cost) - at[g]);
                    const uint32_t begun = classes[g] & __ballot_sync(0xFFFFFFFFu, start <= cost);
                    if (begun == 0u) return 0;
                    const int c = 31 - __clz(begun);
                    return min(rows[g].off[c] + max(0, cost - __shfl_sync(0xFFFFFFFFu, start, c) - kClassRows), rows[g].off[c + 1]);
                };
                const int lo = place(at[NG] * warp / kWarps), hi = warp == kWarps - 1 ? regular_rows[g] : place(at[NG] * (warp + 1) / kWarps);
                if (lo < hi)
                    lbs_regular<NS>(Wb, stride, rows[g], lo, hi, skip[g], s32, ring + warp * kRing * 32, cells + g * 2 * LbsCells<NS>::kWords,
                                    sums + g * 2 * kLbsGroupSums);
            }
        }
    }
    __syncthreads();
}

// V(group, slot k replaced by a channel of score sx): kept sum Ax of the channel, displaced sums D of the other slots.  A slot q is
// among the two leading slots of the three that stay, and so kept unless displaced, where it is among the first two of all four or
// third with k not last (`sums`: M and H, above).
__device__ __forceinline__ double lbs_value(int k, unsigned long long Ax, double sx, const unsigned long long (&D)[3], const unsigned long long *sums,
                                            const double *s) {
    double t[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int qi = q < k ? q : q - 1;
        unsigned long long A = Ax;
        if (q != k) {
            A = sums[12 + q] - (qi == 0 ? D[0] : qi == 1 ? D[1] : D[2]);
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (p != q && p != k) A += sums[lbs_third(q, p)];
        }
        t[q] = __dmul_rn(q == k ? sx : s[q], __dmul_rn(__ll2double_rn((long long)A), 0x1p-24));
    }
    return __dadd_rn(__dadd_rn(__dadd_rn(t[0], t[1]), t[2]), t[3]);
}
__device__ __forceinline__ double lbs_group_value(const unsigned long long (&A)[4], const double *s) {
    double t[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) t[q] = __dmul_rn(s[q], __dmul_rn(__ll2double_rn((long long)A[q]), 0x1p-24));
    return __dadd_rn(__dadd_rn(__dadd_rn(t[0], t[1]), t[2]), t[3]);
}

// Scores of a block's channels into shared memory (zero beyond m), then a barrier.
__device__ __forceinline__ void lbs_load_scores(const double *__restrict__ score, const int32_t *__restrict__ theta0, int p0, int m, double *s64,
                                                float *s32) {
    for (int x = threadIdx.x; x < kLbsMax; x += blockDim.x) {
        const double s = x < m ? score[theta0[p0 + x]] : 0.0;
        s64[x] = s;
        s32[x] = (float)s;
    }
    __syncthreads();
}

// Ascending bitonic sort of the first WIDTH (a power of two, 8 or more) of a warp's 256 non-negative values, eight per lane; the others are zero.
template <int WIDTH>
__device__ __forceinline__ void lbs_sort(float (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= WIDTH; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 8) {
                const bool up = k == 256 || (lane & (k >> 3)) == 0, low = (lane & (j >> 3)) == 0;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float o = __shfl_xor_sync(0xFFFFFFFFu, v[e], j >> 3);
                    v[e] = up == low ? fminf(v[e], o) : fmaxf(v[e], o);
                }
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    if (e & j) continue;
                    const bool up = k >= 8 ? k == 256 || (lane & (k >> 3)) == 0 : (e & k) == 0;
                    const float lo = fminf(v[e], v[e | j]), hi = fmaxf(v[e], v[e | j]);
                    v[e] = up ? lo : hi;
                    v[e | j] = up ? hi : lo;
                }
            }
        }
    }
}

// Hands block b to the exact kernels (again: nothing happens).
__device__ __forceinline__ void lbs_hand_over(int b, int *handed, int *handed_list, unsigned long long *counters) {
    if (atomicExch(&handed[b], 1) == 0) handed_list[atomicAdd(&counters[4], 1ULL)] = b;
}

// Wb[b][row][x] = |W[row, channel x of block b]| bits, `stride` (lbs_block rounded up to 8) per row, zeros beyond the block: one pass over W, permuted
// through shared memory, so that everything below reads whole contiguous rows.  A warp per (row, block). widest[b] becomes the bits of the block's largest
// magnitude, live[b][x] is set where the column of channel x holds anything but zeros; handed[b] is set where the bounds of lbs_bounds.cuh do not hold: a
// weight that is not finite, a score that is neither zero nor of ordinary magnitude, scores more than 2^200 apart; in all of them if `all` says so.
__global__ void __launch_bounds__(256) lbs_gather_kernel(const __half *__restrict__ W, int No, int C, long ldw, const double *__restrict__ score,
                                                         const int32_t *__restrict__ theta0, int lbs_block, int stride, int nblocks,
                                                         int rows_per_cta, uint16_t *__restrict__ Wb, int *__restrict__ handed, int *__restrict__ widest,
                                                         uint8_t *__restrict__ live, bool all, int *__restrict__ handed_list,
                                                         unsigned long long *__restrict__ counters) {
    extern __shared__ __align__(16) uint16_t s_rows[];            // [rows_per_cta][C]
    const int j0 = blockIdx.x * rows_per_cta;
    const int nrows = min(rows_per_cta, No - j0);
    const int per_row = C / 8;
    for (int i = threadIdx.x; i < nrows * per_row; i += 256) {
        const int r = i / per_row, c = (i - r * per_row) * 8;
        uint4 v = __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const uint16_t *>(W) + (long)(j0 + r) * ldw + c));
        v.x &= 0x7FFF7FFFu; v.y &= 0x7FFF7FFFu; v.z &= 0x7FFF7FFFu; v.w &= 0x7FFF7FFFu;
        *reinterpret_cast<uint4 *>(s_rows + (size_t)r * C + c) = v;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, x0 = lane * 8;
    for (int b = threadIdx.x >> 5; b < nblocks; b += 8) {
        const int p0 = b * lbs_block, m = min(lbs_block, C - p0);
        int ch[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) ch[e] = x0 + e < m ? theta0[p0 + x0 + e] : -1;
        bool bad = all;
        if (blockIdx.x == 0) {                                    // the scores, by one CTA (by each, 512 x 36864 in blocks of 8 took 3.70 ms here, 1.74 so)
            int top = -100000, low = 100000;                      // their exponents
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                if (ch[e] < 0) continue;
                const double s = score[ch[e]];
                const bool ordinary = fabs(s) >= 0x1p-300 && fabs(s) <= 0x1p300;
                bad = bad || !(ordinary || s == 0.0);
                if (ordinary) { top = max(top, ilogb(s)); low = min(low, ilogb(s)); }
            }
            top = __reduce_max_sync(0xFFFFFFFFu, top);            // (all lanes, whatever they have found)
            low = __reduce_min_sync(0xFFFFFFFFu, low);
            bad = __any_sync(0xFFFFFFFFu, bad) || top - low > 200;
        }
        uint16_t most[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int r = 0; r < nrows; ++r) {
            uint16_t h[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                h[e] = ch[e] >= 0 ? s_rows[(size_t)r * C + ch[e]] : (uint16_t)0;
                most[e] = max(most[e], h[e]);
            }
            if (x0 < stride)
                *reinterpret_cast<uint4 *>(Wb + ((size_t)b * No + j0 + r) * stride + x0) =
                    make_uint4(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16), h[4] | ((uint32_t)h[5] << 16), h[6] | ((uint32_t)h[7] << 16));
        }
        uint32_t wide = 0, on[2] = {0, 0};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            wide = max(wide, (uint32_t)most[e]);
            on[e >> 2] |= (most[e] ? 1u : 0u) << (8 * (e & 3));
        }
        uint2 *live_at = reinterpret_cast<uint2 *>(live + (size_t)b * stride + x0);
        if (on[0] == 0x01010101u && on[1] == 0x01010101u) *live_at = make_uint2(on[0], on[1]);      // (every CTA that writes a byte writes a one)
        else {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (most[e]) reinterpret_cast<uint8_t *>(live_at)[e] = 1;
        }
        wide = __reduce_max_sync(0xFFFFFFFFu, wide);
        if (lane == 0) atomicMax(&widest[b], (int)wide);
        if ((bad || wide >= 0x7C00u) && lane == 0) lbs_hand_over(b, handed, handed_list, counters);
    }
}

// For the exact kernels: irregular[b][row] is set where the row holds a magnitude of 0.5 or more, or two products that fp32 cannot tell apart (found by
// sorting the row's products: about 700 instructions per row of a 256-channel block; a narrow block sorts no wider than it is -- 512 blocks of
// 8 channels of a 4096 x 4096 weight 2.8 -> 0.77 ms), or the block a score that is no ordinary positive number.  A warp per row of a block.
template <int WIDTH>                                              // lbs_block or more
__global__ void __launch_bounds__(256) lbs_mark_kernel(const uint16_t *__restrict__ Wb, int No, int stride, const double *__restrict__ score,
                                                       const int32_t *__restrict__ theta0, int C, int lbs_block, const int *__restrict__ handed,
                                                       uint8_t *__restrict__ irregular) {
    const int b = blockIdx.y, p0 = b * lbs_block, m = min(lbs_block, C - p0);
    grid_dependency_wait();
    if (!handed[b]) return;
    const int lane = threadIdx.x & 31, x0 = lane * 8;
    float s32[8];
    bool bad = false;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const double s = x0 + e < m ? score[theta0[p0 + x0 + e]] : 1.0;
        s32[e] = (float)s;
        bad = bad || !(s >= 0x1p-80 && s <= 0x1p80);
    }
    bad = __any_sync(0xFFFFFFFFu, bad);
    for (int j = blockIdx.x * 8 + (threadIdx.x >> 5); j < No; j += gridDim.x * 8) {
        const size_t row = (size_t)b * No + j;
        const uint4 v = x0 < stride ? __ldg(reinterpret_cast<const uint4 *>(Wb + row * stride + x0)) : make_uint4(0u, 0u, 0u, 0u);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        uint16_t top = 0;
        float p[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const uint16_t h = (uint16_t)(w[e >> 1] >> (16 * (e & 1)));
            top = max(top, h);
            p[e] = __half2float(__ushort_as_half(h)) * s32[e];
        }
        bool irr = bad || __any_sync(0xFFFFFFFFu, top >= kWideBits);
        if (!irr) {
            lbs_sort<WIDTH>(p);
            float above = __shfl_down_sync(0xFFFFFFFFu, p[0], 1);
            if (lane == 31) above = INFINITY;
            bool close = false;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float hi = e < 7 ? p[e + 1] : above;
                close = close || (hi > 0.f && !(hi - p[e] > hi * kLbsMargin) && hi < INFINITY);
            }
            irr = __any_sync(0xFFFFFFFFu, close);
        }
        if (lane == 0) irregular[row] = irr ? 1 : 0;
    }
}

// Wt[c][row] = |W[row, c]| bits, ldt apart: what a group's own channels are read from (lbs_prepare).  64 x 64 tiles, 16-byte pieces both ways.
__global__ void __launch_bounds__(256) lbs_transpose_kernel(const __half *__restrict__ W, int No, int C, long ldw, uint16_t *__restrict__ Wt, long ldt) {
    __shared__ uint32_t s[64][33];           // [channel][row pair], one word of padding per row
    uint16_t *s16 = reinterpret_cast<uint16_t *>(&s[0][0]);
    const int c0 = blockIdx.x * 64, r0 = blockIdx.y * 64;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int idx = threadIdx.x + 256 * j, piece = idx & 7, row = idx >> 3, c = c0 + piece * 8;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (r0 + row < No && c < C) v = __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const uint16_t *>(W) + (long)(r0 + row) * ldw + c));
        const uint32_t w[4] = {v.x & 0x7FFF7FFFu, v.y & 0x7FFF7FFFu, v.z & 0x7FFF7FFFu, v.w & 0x7FFF7FFFu};
#pragma unroll
        for (int i = 0; i < 8; ++i) s16[(piece * 8 + i) * 66 + row] = (uint16_t)(w[i >> 1] >> (16 * (i & 1)));
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int idx = threadIdx.x + 256 * j, piece = idx & 7, ch = idx >> 3;
        if (c0 + ch < C && r0 + piece * 8 < ldt)
            *reinterpret_cast<uint4 *>(Wt + (long)(c0 + ch) * ldt + r0 + piece * 8) =
                make_uint4(s[ch][piece * 4], s[ch][piece * 4 + 1], s[ch][piece * 4 + 2], s[ch][piece * 4 + 3]);
    }
}

// table[b][g][slot][x] = V(group g of block b with its slot replaced by block channel x); base[G] = V(g).  handed_pos: null = the order theta0.
// One CTA per (block, group of a full block), all rows in chunks.  Two CTAs per SM (128 registers), so that one's sort runs under the other's
// candidates.
constexpr int kTableRows = 1024, kTableThreads = 256;
struct LbsTableSmem {
    LbsRows<kTableRows> rows;
    uint4 ring[kTableThreads / 32 * kRing * 32];
    uint32_t cells[2 * LbsCells<4>::kWords];
    uint32_t sums[2 * kLbsGroupSums];
    unsigned long long total[kLbsGroupSums];
    LbsGroup grp;
    double s64[kLbsMax];
    float s32[kLbsMax];
    int skip;
};
__global__ void __launch_bounds__(kTableThreads, 2) lbs_table_kernel(const uint16_t *__restrict__ Wb, const uint16_t *__restrict__ Wt, long ldt,
                                                                     const uint8_t *__restrict__ irregular, int No, int stride,
                                                                     const double *__restrict__ score, const int32_t *__restrict__ theta0, int C,
                                                                     int lbs_block, const int *__restrict__ handed, const int32_t *__restrict__ handed_pos,
                                                                     double *__restrict__ table, double *__restrict__ base) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    LbsTableSmem &S = *reinterpret_cast<LbsTableSmem *>(s_dyn);
    const int g = blockIdx.x, b = blockIdx.y;
    const int p0 = b * lbs_block, m = min(lbs_block, C - p0);
    grid_dependency_wait();
    if (g * 4 >= m || !handed[b]) return;
    const int tid = threadIdx.x;
    for (int i = tid; i < 2 * LbsCells<4>::kWords; i += kTableThreads) S.cells[i] = 0u;
    if (tid < 2 * kLbsGroupSums) S.sums[tid] = 0u;
    if (tid < 32) S.rows.cnt[tid] = 0;
    lbs_load_scores(score, theta0, p0, m, S.s64, S.s32);
    if (tid < 4) {
        const int x = handed_pos ? handed_pos[p0 + g * 4 + tid] : g * 4 + tid;
        S.grp.channel[tid] = theta0[p0 + x];
        S.grp.s[tid] = S.s64[x];
        S.grp.s32[tid] = S.s32[x];
    }
    if (tid == 0) S.skip = -1;
    __syncthreads();
    const uint16_t *Wblk = Wb + (size_t)b * No * stride;
    const uint8_t *iblk = irregular + (size_t)b * No;
    const int chunk_rows = lbs_chunk_rows(No, kTableRows);
    for (int r0 = 0; r0 < No; r0 += chunk_rows)
        lbs_chunk<1, kTableRows, kTableThreads, 4>(Wblk + (size_t)r0 * stride, stride, Wt + r0, ldt, iblk + r0, min(chunk_rows, No - r0), &S.grp, &S.skip,
                                                   &S.rows, S.s32, S.s64, S.ring, S.cells, S.sums);
    if (tid < kLbsGroupSums) S.total[tid] = lbs_cell(S.sums + tid, kLbsGroupSums);
    __syncthreads();
    const int x = (tid & 31) * 8 + (tid >> 5);                    // cell tid belongs to this candidate
    static_assert(kTableThreads == kLbsMax, "one candidate per thread");
    if (x < m) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            unsigned long long D[3];
#pragma unroll
            for (int qi = 0; qi < 3; ++qi) D[qi] = lbs_cell(S.cells + (4 + 3 * k + qi) * kLbsMax + tid, LbsCells<4>::kWords);
            const unsigned long long A = lbs_cell(S.cells + k * kLbsMax + tid, LbsCells<4>::kWords);
            table[(((long)b * kLbsGroups + g) * 4 + k) * kLbsMax + x] = lbs_value(k, A, S.s64[x], D, S.total, S.grp.s);
        }
    }
    if (tid == 0) {
        const unsigned long long A[4] = {S.total[12], S.total[13], S.total[14], S.total[15]};
        base[p0 / 4 + g] = lbs_group_value(A, S.grp.s);
    }
}

// One cluster of CTAs per block of positions: repeat { best cross-group swap; apply if its gain is positive; refresh the two
// touched groups }.
//   * The output rows are dealt to the CTAs of the cluster: each sorts and sums its own slice for both groups, then each combines
//     an equal share of the (group, slot, candidate) sums of all CTAs through distributed shared memory and writes the table entries.
//     (Dealing candidates instead makes every CTA rank every row: a quarter more work.)
//   * The gains of all position pairs stay in shared memory, pair (i, j) in the CTA of rank i mod cluster size: a swap changes the
//     gains of 8 of the 256 positions, so about 2000 pairs are looked up again in the table (L2) and the search itself reads
//     shared memory only.
// Every CTA takes the same decision from the exchanged winners; all cluster barriers are reached by all threads.
// The i-th cluster takes the i-th block that was handed over, if these are more than `from` and at most `to`.
constexpr int kGreedyRows = 1024, kGreedyThreads = 512, kGreedyMaxCluster = 16, kGreedyMinCluster = 3;
constexpr int kLbsSwapLimit = 1 << 16;                            // far above any block's swaps; beyond it the kernel reports a timeout
struct LbsGreedySmem {
    uint32_t cells[2][2 * LbsCells<3>::kWords];
    LbsRows<kGreedyRows> rows[2];
    uint4 ring[kGreedyThreads / 32 * kRing * 32];
    uint32_t sums[2][2 * kLbsGroupSums];
    unsigned long long total[2][kLbsGroupSums];                   // `sums` over all CTAs of the cluster
    LbsGroup grp[2];
    double s64[kLbsMax];
    float s32[kLbsMax];
    int pos2x[kLbsMax], chan[kLbsMax];
    double base[kLbsGroups];
    double red_gain[kGreedyThreads / 32], red_second[kGreedyThreads / 32];
    int red_at[kGreedyThreads / 32];
    double won_gain[kGreedyMaxCluster], won_second[kGreedyMaxCluster];      // written by the CTAs of the cluster
    int won_pair[kGreedyMaxCluster];
    int skip[2];
    double gains[1];                                              // [local rows] of m - 1 - i pairs each
};
// Pairs (i, j > i) held by one CTA: rows i = rank, rank + nc, ..., one after the other (so places ascend with (i, j)).
__host__ __device__ inline int lbs_gain_offset(int r, int m, int rank, int nc) { return r * (m - 1 - rank) - nc * (r * (r - 1) / 2); }
inline size_t lbs_greedy_smem(int nc) { return sizeof(LbsGreedySmem) + sizeof(double) * (size_t)lbs_gain_offset((kLbsMax + nc - 1) / nc, kLbsMax, 0, nc); }

__device__ __forceinline__ long long lbs_order_key(double v) {    // ascending as a signed integer
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFLL);
}
__device__ __forceinline__ double lbs_warp_max(double v, int &hi, uint32_t &lo) {
    const long long k = lbs_order_key(v);
    hi = __reduce_max_sync(0xFFFFFFFFu, (int)(k >> 32));
    lo = __reduce_max_sync(0xFFFFFFFFu, (int)(k >> 32) == hi ? (uint32_t)k : 0u);
    const long long top = ((long long)hi << 32) | lo;
    return __longlong_as_double(top ^ ((top >> 63) & 0x7FFFFFFFFFFFFFFFLL));
}
// (best, second, id) of the warp's 32 entries: the largest best (ties: smallest id), and the largest gain once one instance of it is
// set aside.  Integer reductions of the two halves of an order-preserving key instead of rounds of shuffled doubles.
__device__ __forceinline__ void lbs_warp_best(double &best, double &second, int &id) {
    int hi;
    uint32_t lo;
    const double top = lbs_warp_max(best, hi, lo);
    const long long k = lbs_order_key(best);
    const bool win = (int)(k >> 32) == hi && (uint32_t)k == lo;
    const int first = (int)__reduce_min_sync(0xFFFFFFFFu, win ? (uint32_t)id : 0xFFFFFFFFu);
    second = lbs_warp_max(win && id == first ? second : best, hi, lo);
    best = top;
    id = first;
}
__device__ __forceinline__ void st_remote_f64(uint32_t remote_addr, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote_addr), "d"(v) : "memory");
}
__device__ __forceinline__ void st_remote_s32(uint32_t remote_addr, int v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(remote_addr), "r"(v) : "memory");
}
// A cell summed over the CTAs of the cluster.
__device__ __forceinline__ unsigned long long lbs_cluster_cell(const uint32_t *cell, int n, int nc) {
    const uint32_t at = smem_u32(cell);
    unsigned long long v = 0;
    for (int c0 = 0; c0 < nc; c0 += 8) {     // (sixteen loads in flight)
        uint32_t lo[8], hi[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            lo[c] = hi[c] = 0u;
            if (c0 + c < nc) {
                const uint32_t remote = map_to_rank(at, (uint32_t)(c0 + c));
                asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(lo[c]) : "r"(remote));
                asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(hi[c]) : "r"(remote + 4u * (uint32_t)n));
            }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) v += ((unsigned long long)hi[c] << 32) | lo[c];
    }
    return v;
}

__global__ void __launch_bounds__(kGreedyThreads, 1) lbs_greedy_kernel(const uint16_t *__restrict__ Wb, const uint16_t *__restrict__ Wt, long ldt,
                                                                       const uint8_t *__restrict__ irregular, int No, int stride,
                                                                       const double *__restrict__ score, const int32_t *__restrict__ theta0, int C,
                                                                       int lbs_block, int max_swaps, double *__restrict__ table,
                                                                       const double *__restrict__ base0, int32_t *__restrict__ theta,
                                                                       unsigned long long *__restrict__ counters, const int *__restrict__ handed_list,
                                                                       const int *__restrict__ handed_swaps, const int32_t *__restrict__ handed_pos, int nc,
                                                                       int from, int to) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    LbsGreedySmem &S = *reinterpret_cast<LbsGreedySmem *>(s_dyn);
    using Cells = LbsCells<3>;
    const int number = (int)counters[4], at_list = blockIdx.x / nc;
    if (number <= from || number > to || at_list >= number) return;
    const int b = handed_list[at_list], rank = (int)cluster_ctarank();
    const int p0 = b * lbs_block, m = min(lbs_block, C - p0), G = m / 4;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int kWarps = kGreedyThreads / 32;
    double *tb = table + (long)b * kLbsGroups * 4 * kLbsMax;      // row of position i: group i / 4, slot i % 4
    auto clear_sums = [&]() {
        for (int i = tid; i < (int)(sizeof(S.cells) / 16); i += kGreedyThreads) reinterpret_cast<uint4 *>(S.cells)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (tid < 4 * kLbsGroupSums) (&S.sums[0][0])[tid] = 0u;
    };
    clear_sums();
    if (tid < 64) S.rows[tid >> 5].cnt[tid & 31] = 0;
    for (int x = tid; x < m; x += kGreedyThreads) { S.pos2x[x] = handed_pos ? handed_pos[p0 + x] : x; S.chan[x] = theta0[p0 + x]; }
    for (int g = tid; g < G; g += kGreedyThreads) S.base[g] = base0[p0 / 4 + g];
    lbs_load_scores(score, theta0, p0, m, S.s64, S.s32);          // (ends with a barrier: everything above is visible)
    const int per_cta = (No + nc - 1) / nc, row0 = min(No, rank * per_cta), nrows_all = min(No, row0 + per_cta) - row0, chunk_rows = lbs_chunk_rows(nrows_all, kGreedyRows);
    const uint16_t *Wblk = Wb + ((size_t)b * No + row0) * stride;
    const uint8_t *iblk = irregular + (size_t)b * No + row0;

    // rows of the table are rewritten by other CTAs of the cluster: read from L2, never from this SM's L1
    const int my_rows = rank < m ? (m - rank + nc - 1) / nc : 0, my_pairs = lbs_gain_offset(my_rows, m, rank, nc);
    for (int r = warp; r < my_rows; r += kWarps) {
        const int i = rank + nc * r;
        double *gr = S.gains + lbs_gain_offset(r, m, rank, nc);
#pragma unroll 4
        for (int j = i + 1 + lane; j < m; j += 32) {
            const double after = __dadd_rn(__ldcg(&tb[i * kLbsMax + S.pos2x[j]]), __ldcg(&tb[j * kLbsMax + S.pos2x[i]]));
            gr[j - i - 1] = (i >> 2) == (j >> 2) ? -INFINITY : __dsub_rn(after, __dadd_rn(S.base[i >> 2], S.base[j >> 2]));
        }
    }
    // (a barrier of the cluster, not of the CTA: the first exchange below stores into the shared memory of the other CTAs, which have to be
    // running by then)
    cluster_arrive();
    cluster_wait();
    const int swaps0 = handed_swaps[b];
    int swaps = swaps0, near_swaps = 0;
    for (;;) {
        double best = -INFINITY, second = -INFINITY;              // second: largest gain once one instance of the best is set aside
        int at = 0x7FFFFFFF;
        if (max_swaps <= 0 || swaps < max_swaps) {
#pragma unroll 4
            for (int t = tid; t < my_pairs; t += kGreedyThreads) {
                const double gain = S.gains[t];
                const bool up = gain > best;
                second = up ? best : gain > second ? gain : second;
                best = up ? gain : best;
                at = up ? t : at;
            }
        }
        lbs_warp_best(best, second, at);
        if (lane == 0) { S.red_gain[warp] = best; S.red_second[warp] = second; S.red_at[warp] = at; }
        __syncthreads();
        if (warp == 0) {
            best = lane < kWarps ? S.red_gain[lane] : -INFINITY;
            second = lane < kWarps ? S.red_second[lane] : -INFINITY;
            at = lane < kWarps ? S.red_at[lane] : 0x7FFFFFFF;
            lbs_warp_best(best, second, at);
            int pair = 0x7FFFFFFF;
            int r = -1;                                           // the row that place `at` lies in
#pragma unroll
            for (int q = 0; q < (kLbsMax / kGreedyMinCluster + 32) / 32; ++q) {
                const int row = q * 32 + lane;
                r += __popc(__ballot_sync(0xFFFFFFFFu, row < my_rows && lbs_gain_offset(row, m, rank, nc) <= at));
            }
            if (at != 0x7FFFFFFF) {
                const int i = rank + nc * r;
                pair = i * kLbsMax + at - lbs_gain_offset(r, m, rank, nc) + i + 1;
            }
            if (lane < nc) {                                      // this CTA's winner to every CTA of the cluster
                st_remote_f64(map_to_rank(smem_u32(&S.won_gain[rank]), (uint32_t)lane), best);
                st_remote_f64(map_to_rank(smem_u32(&S.won_second[rank]), (uint32_t)lane), second);
                st_remote_s32(map_to_rank(smem_u32(&S.won_pair[rank]), (uint32_t)lane), pair);
            }
        }
        cluster_arrive();
        cluster_wait();
        best = lane < nc ? S.won_gain[lane] : -INFINITY;
        second = lane < nc ? S.won_second[lane] : -INFINITY;
        int pair = lane < nc ? S.won_pair[lane] : 0x7FFFFFFF;
        lbs_warp_best(best, second, pair);                        // (every warp, the same result: no further exchange)
        if (!(best > 0.0)) break;
        if (second > -INFINITY && __dsub_rn(best, second) < __dmul_rn(1e-6, fabs(best))) ++near_swaps;      // counted, not acted on
        if (++swaps > kLbsSwapLimit) {
            if (tid == 0) atomicExch(&g_device_status, (int)ESP_ERR_TIMEOUT);
            break;
        }
        const int bi = pair >> 8, bj = pair & 255, ga = bi >> 2, gb = bj >> 2;
        const int xi = S.pos2x[bi], xj = S.pos2x[bj];             // (the channels that change places)
        if (tid < 8) {
            const int which = tid >> 2, k = tid & 3, p = (which ? gb : ga) * 4 + k, x = p == bi ? xj : p == bj ? xi : S.pos2x[p];
            S.grp[which].channel[k] = S.chan[x];
            S.grp[which].s[k] = S.s64[x];
            S.grp[which].s32[k] = S.s32[x];
            if (k == 0) S.skip[which] = (which ? bj : bi) & 3;
        }
        if (tid == 32 && rank == 0) {     // the row of a swapped slot now offers the channel that left it: the group as it was
            tb[bi * kLbsMax + xi] = S.base[ga];
            tb[bj * kLbsMax + xj] = S.base[gb];
        }
        __syncthreads();
        if (tid == 0) { S.pos2x[bi] = xj; S.pos2x[bj] = xi; }
        // Row (g, slot) of the table holds g with that slot replaced, so it depends on g's OTHER three channels: the rows of the two
        // swapped slots stay as they are (but for the channel that left them, which was no candidate before).
        for (int r0 = 0; r0 < nrows_all; r0 += chunk_rows)
            lbs_chunk<2, kGreedyRows, kGreedyThreads, 3>(Wblk + (size_t)r0 * stride, stride, Wt + row0 + r0, ldt, iblk + r0, min(chunk_rows, nrows_all - r0),
                                                         S.grp, S.skip, S.rows, S.s32, S.s64, S.ring, &S.cells[0][0], &S.sums[0][0]);
        cluster_arrive();
        cluster_wait();                                           // the sums of every CTA are complete
        constexpr int kEntries = 2 * 3 * kLbsMax;                 // (group, live slot, candidate); this CTA finishes `share` of them
        const int share = ((kEntries + nc - 1) / nc + 31) & ~31, e0 = rank * share;
        unsigned long long *part = reinterpret_cast<unsigned long long *>(S.rows);      // [4 sums][share]: the sorted rows are used up
        static_assert(sizeof(S.rows[0].rec) >= 4 * 8 * (kEntries / kGreedyMinCluster), "room for the largest share, counters untouched");
        if (tid >= kGreedyThreads - 2 * kLbsGroupSums) {          // (the last warp: the fewest entries below are its own)
            const int t = tid - (kGreedyThreads - 2 * kLbsGroupSums);
            S.total[t / kLbsGroupSums][t % kLbsGroupSums] = lbs_cluster_cell(&S.sums[t / kLbsGroupSums][t % kLbsGroupSums], kLbsGroupSums, nc);
        }
        for (int t = tid; t < 4 * share; t += kGreedyThreads) {
            const int sel = t / share, e = e0 + t - sel * share;
            if (e < kEntries) {
                const int which = e / (3 * kLbsMax), live = (e / kLbsMax) % 3, c = e % kLbsMax;
                part[t] = lbs_cluster_cell(&S.cells[which][(sel == 0 ? live : 2 + live * 3 + sel) * kLbsMax + c], Cells::kWords, nc);
            }
        }
        __syncthreads();
        for (int t = tid; t < share; t += kGreedyThreads) {
            const int e = e0 + t;
            if (e >= kEntries) break;
            const int which = e / (3 * kLbsMax), live = (e / kLbsMax) % 3, c = e % kLbsMax, x = (c & 31) * 8 + (c >> 5);
            const int k = live + (live >= S.skip[which] ? 1 : 0);
            const unsigned long long D[3] = {part[share + t], part[2 * share + t], part[3 * share + t]};
            if (x < m) tb[((which ? gb : ga) * 4 + k) * kLbsMax + x] = lbs_value(k, part[t], S.s64[x], D, S.total[which], S.grp[which].s);
        }
        if (tid < 2) {
            const unsigned long long *T = S.total[tid] + 12, A[4] = {T[0], T[1], T[2], T[3]};
            S.base[tid == 0 ? ga : gb] = lbs_group_value(A, S.grp[tid].s);
        }
        __threadfence();
        cluster_arrive();
        cluster_wait();                                           // the new table rows are written, the sums have been read
        // the pairs of the eight positions of both groups: all lookups in flight together
        constexpr int kPer = 8 * kLbsMax / kGreedyThreads;
        double there[kPer], back[kPer];
        int place[kPer];
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int t = tid + u * kGreedyThreads, which = t >> 8, p = (which < 4 ? ga : gb) * 4 + (which & 3), q = t & 255;
            const int i = min(p, q), j = max(p, q);
            place[u] = -1;
            if (j < m && (i >> 2) != (j >> 2) && i % nc == rank) {
                place[u] = i * kLbsMax + j;
                there[u] = __ldcg(&tb[i * kLbsMax + S.pos2x[j]]);
                back[u] = __ldcg(&tb[j * kLbsMax + S.pos2x[i]]);
            }
        }
        clear_sums();
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            if (place[u] < 0) continue;
            const int i = place[u] >> 8, j = place[u] & 255;
            S.gains[lbs_gain_offset((i - rank) / nc, m, rank, nc) + j - i - 1] =
                __dsub_rn(__dadd_rn(there[u], back[u]), __dadd_rn(S.base[i >> 2], S.base[j >> 2]));
        }
        __syncthreads();
    }
    if (rank != 0) return;
    for (int x = tid; x < m; x += kGreedyThreads) theta[p0 + x] = S.chan[S.pos2x[x]];
    if (tid == 0 && swaps > swaps0) atomicAdd(&counters[1], (unsigned long long)(swaps - swaps0));
    if (tid == 0 && near_swaps) atomicAdd(&counters[3], (unsigned long long)near_swaps);
}

inline void lbs_greedy_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr, int nblocks, int nc, cudaStream_t stream) {
    cfg = {};
    cfg.gridDim = dim3(nblocks * nc);
    cfg.blockDim = dim3(kGreedyThreads);
    cfg.dynamicSmemBytes = lbs_greedy_smem(nc);
    cfg.stream = stream;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = nc;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
}

#include "lbs_bounds.cuh"
