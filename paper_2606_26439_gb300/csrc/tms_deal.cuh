// tms_deal.cuh -- which CTA scores which candidates of per-query lists.
//
// The flat list of all queries' candidates is cut into one part per CTA, so a
// CTA meets a few queries only: it loads few query tiles (tables) and leaves
// few super-tiles part empty.  Within a query, the CTAs that meet it take its
// candidates in turn (Columns), so that neighbours in the list, often alike in
// length, are spread over them.
//
// Parts of equal count are parts of equal work while all lists draw their
// documents from the same lengths.  A batch over short and long passages is
// not like that: one list of 180-token documents and fifteen of 32-token ones,
// 10,000 each, took 598 us (fp16) and 595 (FP8) in parts of equal count,
// because the long list's CTAs finished last; every query dealt to every CTA,
// which balances any lists, took 337 and 296.  So a few candidates of each list
// are sampled first, the same ones by every CTA, and where a list's documents
// are longer than the average by a quarter, the parts are of equal estimated
// work: 232 and 199.  Like lists keep parts of equal count, whose balance no
// estimate reaches, and pay 0.5 to 1.5 us (16 x 1,000, fp16: 66.2 and 66.8).  The
// PQ kernel has no spare bandwidth to make up for uneven parts: the same lists
// of 30,000, fp32 table, took 5,387 us in parts of equal count (2,952 with every
// query dealt to every CTA), now 2,052.
#pragma once

#include "tms_common.cuh"

namespace tms {

namespace deal {

constexpr int kGroups = 32;   // lists told apart, one per lane; more are taken as groups of consecutive ones
constexpr int kSums = 32;     // sums of 32 samples each: four for each of up to 8 groups, two for up to 16, else one

struct Lists {
    const int64_t* offsets;  // [n_queries + 1]
    const int32_t* ids;
    const int32_t* lengths;
    int64_t n_docs;
    int n_queries;
    int total;  // entries of ids
};

__device__ __forceinline__ int bound(const Lists& l, int i) {
    const int64_t x = __ldg(l.offsets + i);
    return static_cast<int>(x < 0 ? 0 : (x > l.total ? l.total : x));
}

// The groups, which cover all entries in order; lane g < count has group g.
struct Groups {
    int count, sums;  // sums of each: 1 << sums
    int first, n;     // this lane's entries; n < 0: not a valid list

    __device__ __forceinline__ explicit Groups(const Lists& l) : count(min(l.n_queries, kGroups)) {
        const int lane = threadIdx.x & 31;
        sums = count <= 8 ? 2 : (count <= 16 ? 1 : 0);
        first = lane > 0 && lane < count ? bound(l, lane * l.n_queries / count) : 0;
        const int next = __shfl_down_sync(0xffffffffu, first, 1);
        n = lane < count ? (lane == count - 1 ? l.total : next) - first : 0;
    }
};

// Sums of 32 sampled candidates' rows each (rounded up to UNIT rows per
// document, and DOC more for what it costs beside them), to sums[kSums] in
// shared memory; the warps share the work.  The
// samples are runs of eight neighbours, evenly spaced: a scattered load takes a
// cycle for each of its lines, and twice as many samples of a place each took
// 3 us.  Two loads, one after the other, whatever the lists.
template <int UNIT, int DOC>
__device__ __forceinline__ void sample(const Lists& l, int* sums, int warp, int warps) {
    constexpr int kBatch = 8;
    const int lane = threadIdx.x & 31;
    const Groups groups(l);
    const int tasks = groups.count << groups.sums;
#pragma unroll 1
    for (int t0 = warp; t0 < tasks; t0 += kBatch * warps) {
        int x[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int t = t0 + b * warps, g = (t >> groups.sums) & 31;
            const int first = __shfl_sync(0xffffffffu, groups.first, g), n = __shfl_sync(0xffffffffu, groups.n, g);
            const int run = (t & ((1 << groups.sums) - 1)) * 4 + (lane >> 3);  // of 4 << sums
            const int at = static_cast<int>((static_cast<int64_t>(2 * run + 1) * n) >> (3 + groups.sums)) + (lane & 7);
            x[b] = t < tasks && n > 0 ? __ldg(l.ids + first + min(at, n - 1)) : -1;
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) x[b] = x[b] >= 0 && x[b] < l.n_docs ? __ldg(l.lengths + x[b]) : 0;
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int rows = (min(max(x[b], 0), 1 << 20) + UNIT - 1) & ~(UNIT - 1);
            const int s = __reduce_add_sync(0xffffffffu, rows + DOC);
            if (lane == 0 && t0 + b * warps < tasks) sums[t0 + b * warps] = s;
        }
    }
}

struct Part {
    int lo, hi;   // entries [lo, hi) of the flat list
    bool uneven;  // parts of equal estimated work
};

// In shared memory; what follows it there is aligned to 16 bytes.
struct alignas(16) Shared {
    int sums[kSums];  // of sampled rows; where the parts are uneven, then CTAs per candidate of each group (float)
    Part part;        // uneven false: the parts are of equal count
};
static_assert(sizeof(Shared) % 16 == 0, "the regions after it stay aligned");

// This CTA's part of equal count.
__device__ __forceinline__ Part equal_part(int total) {
    const int grid = gridDim.x, block = blockIdx.x;
    const int each = total / grid, more = total - each * grid;
    auto start = [&](int b) { return each * b + more * b / grid; };  // total * b / grid
    return Part{start(block), start(block + 1), false};
}

// This CTA's part of equal estimated work to sh.part, if the lists are unlike
// enough for it; else sh.part.uneven is false.  One warp, the same outcome in
// every CTA; sh.sums as sample left them.
__device__ __forceinline__ void uneven_part(const Lists& l, Shared& sh) {
    const int lane = threadIdx.x & 31;
    const int grid = gridDim.x;
    const Groups groups(l);
    const int first = groups.first, n = groups.n;
    int s = 0;  // the group's sampled rows
    if (lane < groups.count)
        for (int r = 0; r < 1 << groups.sums; ++r) s += sh.sums[(lane << groups.sums) + r];
    float all = static_cast<float>(n) * static_cast<float>(s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
    // longer documents than the average by a quarter, in a group that is worth
    // half a part or more (lengths uniform on [32, 180]: three standard errors
    // of the mean of 64 samples are 15%)
    const bool longer = n > l.total / grid / 2 && static_cast<float>(s) * static_cast<float>(l.total) > 1.25f * all;
    if (!__any_sync(0xffffffffu, longer) || __any_sync(0xffffffffu, n < 0)) {
        if (lane == 0) sh.part.uneven = false;
        return;
    }
    const unsigned long long w = static_cast<unsigned long long>(n) * static_cast<unsigned>(s);  // estimated work
    unsigned long long end = w;                                                                  // and its prefix
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, end, o);
        if (lane >= o) end += y;
    }
    const unsigned long long work = __shfl_sync(0xffffffffu, end, 31);
    auto place = [&](int b) {  // where the work before part b ends
        if (b == 0 || b == grid) return b == 0 ? 0 : l.total;
        const unsigned long long t = work / grid * b + work % grid * b / grid;
        const int src = 31 - __clz(__ballot_sync(0xffffffffu, w > 0 && end - w <= t));
        const unsigned long long gw = __shfl_sync(0xffffffffu, w, src), ge = __shfl_sync(0xffffffffu, end, src);
        const int gf = __shfl_sync(0xffffffffu, first, src), gn = __shfl_sync(0xffffffffu, n, src);
        const float x = static_cast<float>(t - (ge - gw)) / static_cast<float>(gw) * static_cast<float>(gn);
        return gf + min(gn, static_cast<int>(x));
    };
    const Part p{place(blockIdx.x), place(blockIdx.x + 1), true};
    if (lane == 0) sh.part = p;
    if (lane < groups.count)  // every lane has read the sums before the votes
        sh.sums[lane] = __float_as_int(static_cast<float>(s) * static_cast<float>(grid) / static_cast<float>(work));
}

// Entries [c0, end) of one query, taken in turn by the w or so CTAs that meet
// it: place x of the list is candidate t w + col, the t-th of column col.  The
// first `rem` columns have `tall` entries (`wide` together), the others one
// fewer.
struct Columns {
    int c0, end;
    int w, wide, tall, rem;

    // `parts`: CTAs per candidate, or any number that all CTAs agree on: those
    // of the list's group where the parts are uneven and each group is one list,
    // else of all lists (of many, a CTA or two meet one anyway).
    __device__ __forceinline__ void enter(int first, int last, float parts) {
        c0 = first, end = last;
        if (c0 >= end) return;
        w = min(max(__float2int_rn(static_cast<float>(end - c0) * parts), 1), end - c0);
        tall = (end - c0 + w - 1) / w;
        rem = end - c0 - (tall - 1) * w;
        wide = rem * tall;
    }
    // Column and place in it of place p, c0 <= p < end.
    __device__ __forceinline__ void find(int p, int* col, int* t) const {
        int x = p - c0;
        if (x < wide) {
            *col = x / tall;
            *t = x - *col * tall;
        } else {
            x -= wide;
            *col = x / (tall - 1);
            *t = x - *col * (tall - 1);
            *col += rem;
        }
    }
    __device__ __forceinline__ int entry(int col, int t) const { return c0 + t * w + col; }
    // Entry at place p, c0 <= p < end.
    __device__ __forceinline__ int at(int p) const {
        int col, t;
        find(p, &col, &t);
        return entry(col, t);
    }
    // Entry `more` places on from (col, t), still before end: a part spans a
    // column or two, so this needs no division.
    __device__ __forceinline__ int ahead(int col, int t, int more) const {
        t += more;
        for (int h = col < rem ? tall : tall - 1; t >= h; h = col < rem ? tall : tall - 1) {
            t -= h;
            ++col;
        }
        return entry(col, t);
    }
};

}  // namespace deal

}  // namespace tms
