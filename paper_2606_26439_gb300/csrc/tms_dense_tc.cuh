// tms_dense_tc.cuh -- the tensor-core dense MaxSim kernel and its launcher.
//
// Computes Eq. 1 of the TileMaxSim paper, score = sum_i max_j q_i . d_j,
// for every candidate of every query, in one persistent launch, with the
// document and query rows stored as fp16 / bf16, as FP8 E4M3 codes with one
// fp32 scale per row (F8), or as fp32 scored by split TF32 (TF: each
// operand x = hi + lo with hi = x with its 13 low mantissa bits cleared --
// the value a kind::tf32 MMA reads from an fp32 element -- and lo = x - hi
// exact; hi.hi + hi.lo + lo.hi on the tensor cores, the lo.lo term of
// relative size below 2^-20 dropped -- FP32-level accuracy).
//
// Orientation: the MMA computes S^T = Q D^T, query tokens along M (tensor-
// memory lanes, one per epilogue thread) and document rows along N
// (tensor-memory columns).  The max over a document's tokens (Eq. 1's
// inner max) is then a running max inside each thread's registers -- no
// cross-lane reduction.  M is always 128: the query tile's 32-row blocks
// (token blocks of one query, or the queries of a shared group) are
// replicated down the 128 rows when they are fewer.
//
// Super-tiles: consecutive documents are packed in units of 8 rows, side by
// side, into one super-tile of up to 256 or 128 rows, and one run of MMAs
// (N = the packed rows rounded up to 16) scores them all.  The per-tile
// costs of the pipeline -- barrier round trips, commits, MMA issue -- are
// paid once per super-tile, typically two to three documents.
//
//   * Planner warp: takes the CTA's candidates (Work) 32 at a time, one per
//     lane (metadata, validity, query, -inf / NaN for empty / bad documents),
//     places their units in super-tiles with one scan and publishes each
//     super-tile as one record -- header, tile list, documents that end in
//     it -- with a single barrier arrival.  It also loads each query's tile
//     (replicated, see above).
//   * Loader warp: streams each super-tile from HBM into a ring of shared-
//     memory chunk stages (STR rows x 128 bytes: 64 fp16/bf16 or 128 E4M3
//     elements per row), one TMA box per tile and chunk, the tiles issued
//     by parallel lanes (128-byte swizzle).  Each token is read from HBM
//     once (Theorem 1 with BQ = Nq, or the whole group of queries in the
//     shared schedule).
//   * TF only -- eight splitter warps: split every landed chunk stage (hi in
//     place, lo beside it) before the MMA reads it, and every new query tile
//     that does not lie in tensor memory (see kQueryCols).
//   * Two MMA warps, super-tiles in turn: an elected lane issues tcgen05.mma
//     (M = 128 query rows, K = 32 bytes: 16 fp16/bf16 elements with
//     kind::f16, 32 E4M3 elements with kind::f8f6f4, 8 TF32 elements --
//     three products -- with kind::tf32) over every dimension chunk of a
//     super-tile, accumulating the partial dot products in tensor memory
//     before any max is taken -- the paper's dimension tiling (Section 3),
//     with the K loop running through TMEM.
//   * Epilogue warps (four for each 128-row half): thread = query row (TMEM
//     lane).  Each warp takes its columns of a super-tile with tcgen05.ld,
//     multiplies column j by document row j's scale (F8), and reduces them to
//     a running max that starts again after each document's end.
//   * Shared lists: a warp sees all columns of its query and sums each
//     document's row maxima over the query tokens (times their scales, F8)
//     itself.  Per-query lists: the copies share the columns and leave their
//     values at documents' ends, and at the end of their share, in shared
//     memory; a finisher warp combines and sums them.  Each score is written
//     once; the Nq x Nd similarity matrix never reaches HBM and no atomics or
//     memset are needed.
//
// Every wait is bounded (see tms_common.cuh); a timeout sets
// TMS_DEVERR_TIMEOUT and the CTA drains its in-flight copies and MMAs,
// frees its tensor memory and returns.
#pragma once

#include <algorithm>
#include <map>
#include <mutex>

#include "tms_common.cuh"
#include "tms_deal.cuh"
#include "tms_internal.h"

namespace tms {

namespace dense {

constexpr int kRows = 128;                    // document rows per tile
// Row types: fp16 / bf16, FP8 E4M3 codes + row scales, fp32 by split TF32,
// PQ codes decompressed into fp16 rows in shared memory (kPQ: M = 16
// subspaces of 8 dimensions, d = 128).
enum : int { kF16 = 0, kE4M3 = 1, kTF32 = 2, kPQ = 3 };
// Elements per 128-byte dimension chunk (one 128-byte swizzle row).
__host__ __device__ constexpr int chunk_elems(int kind) { return kind == kE4M3 ? 128 : (kind == kTF32 ? 32 : 64); }
constexpr int kPqM = 16;                      // kPQ: subspaces (16 code bytes per token)
constexpr int kPqCbBytes = 256 * kPqM * 16;   // kPQ: fp16 codebook, all 256 codes (64 KB)
constexpr int kCodeRing = 4;                  // kPQ: super-tiles whose code rows are in flight or held
constexpr int kBoxKinds = kRows / 8;          // box heights 8, 16, ..., 128
constexpr int kMaxSeg = 32;                   // tiles per super-tile (each >= 8 rows, one per planner lane)
// Super-tile records in flight.  A record slot is republished only after
// every role has passed it, so the ring also bounds how far the loader can
// run ahead of the epilogue: with HBM latencies of a few microseconds under
// load, the loads of many super-tiles must be in flight at once: 16 of 128
// rows, 8 of 256.
__host__ __device__ constexpr int st_ring(int str) { return str == 256 ? 8 : 16; }
// Epilogue warps: one per tensor-memory lane quarter and query half.
__host__ __device__ constexpr int epi_warps(int h) { return 4 * h; }
// Warps that prepare every chunk stage.  TF: splitters -- four of them took
// 1,150 cycles per 16 KB stage, against 770 for its MMAs and 670 for its bytes
// from HBM; kPQ: decompressors.
__host__ __device__ constexpr int help_warps(int kind) { return kind == kTF32 ? 8 : 4; }
// Finisher warp, where the copies of a query's blocks share a super-tile's
// columns (per-query lists).
__host__ __device__ constexpr int fin_warps(bool sh) { return sh ? 0 : 1; }
constexpr int kMaxBlocks = 4;  // 32-token blocks of a query
// MMA warps, taking super-tiles in turn: issuing an MMA takes its thread about
// 50 cycles, a commit 64, a wait that need not wait 70 (measured), so beside
// 64- or 128-cycle MMAs one thread cannot keep the tensor core busy.
constexpr int kMmaWarps = 2;
// planner, MMA warps, loader, epilogue warps, finisher, splitters / decompressors
__host__ __device__ constexpr int kernel_threads(int kind, int h, bool sh) {
    return 32 * (2 + kMmaWarps + epi_warps(h) + fin_warps(sh) + ((kind == kTF32 || kind == kPQ) ? help_warps(kind) : 0));
}
// Split TF32 with the query's hi and lo parts in tensor memory as the MMA's A
// operand, where they fit (QT: 32 columns each per 32-element chunk, up to
// kQueryCols): the MMAs, three per K-step over 128 columns, then read 64 B of
// shared memory a cycle instead of 128, beside the fills and the splits of the
// stages (32 B each); the query tile needs no copies and no lo twin in shared
// memory, which leaves room for two more stages.
constexpr int kQueryCols = 256;
constexpr int kQueryChunks = kQueryCols / 64;
// Accumulator buffers of STR tensor-memory columns -- one holds one query
// half of a super-tile -- as many as the SM's 512 columns give the CTAs
// sharing it, at most four.
__host__ __device__ constexpr int acc_count(int str, int ctas, bool qt) {
    const int n = (512 - (qt ? kQueryCols : 0)) / (str * ctas);
    return n < 4 ? n : 4;
}
constexpr int kMaxStages = 16;
// Per-query lists: candidates per CTA from which their lengths are sampled (one
// list of 180-token and fifteen of 32-token documents, 1,000 each, FP8, 52 per
// CTA: 64.6 us not sampled, 29.2 sampled; 16 like lists of 650, 34 per CTA: 38.3
// and 39.5).
constexpr int kMinSampled = 24;
constexpr int kSmemLimit = 232448;            // 227 KB opt-in maximum per CTA

enum : int { kEnd = 1 };

// A super-tile is filled in units of 8 rows, each of one document: a document
// of n tokens takes ceil(n / 8) units, the last of them partial (rows of the
// next document past its end, dropped by the epilogue) if n % 8 != 0.

// One document tile inside a super-tile: consecutive token rows.
struct SegInfo {
    int row0;       // token row of the tile's first row
    uint8_t nu;     // units (1..16)
    uint8_t cu;     // first unit of the super-tile
    uint16_t rows;  // rows that count (8 nu but for a partial last unit)
};

// One super-tile record (planner -> loader, MMA warps and epilogue).
struct StHdr {
    int q;            // query (group) whose tile it is scored against
    int n;            // MMA N: packed rows rounded up to 16
    int nseg;         // tiles
    int flags;        // kEnd
    int rows;         // packed rows: 8 x units
    uint32_t ends;     // bit u: unit u is the last of a document (f[] in that order)
    uint32_t partial;  // bit u: and not all of its rows count
    // per-query lists, bit u: the epilogue leaves a value at unit u, the last of
    // a document, or of a copy's share of the columns where its document goes on
    uint32_t values;
};

struct StSlot {
    StHdr h;
    SegInfo seg[kMaxSeg];
    int f[kMaxSeg];          // documents that end here: flat candidate index (shared mode: position in the list)
    uint8_t valid[kMaxSeg];  // by unit, where a document ends: its rows that count (1..8)
};

struct Args {
    const int64_t* offsets;
    const int32_t* lengths;
    const int32_t* cand_ids;
    const int64_t* cand_offsets;
    float* out;
    const float* q_scales;  // F8: [n_queries * nq] per-query-token scales
    const float* t_scales;  // F8: [n_tokens] per-document-token scales
    unsigned int* err;
    int64_t n_docs;
    int64_t n_tokens;
    int64_t n_cand;    // entries of cand_ids
    int64_t n_flat;    // work items: n_cand, or n_groups * n_cand in shared mode
    int group;         // shared mode: queries per group; 0 otherwise
    int rounds;        // shared mode: see Work; set by launch_tc
    int round_groups;  // groups of every round but the last
    int last_groups;   // groups of the last round
    int n_queries;
    int nq;
    int sampled;     // per-query lists: parts by estimated work (tms_deal.cuh); set by launch_tc
    int nchunks;     // ceil(d / chunk_elems)
    int stages;      // chunk stages in the ring
    int qslots;      // resident query-tile slots; 0: the query is streamed with each chunk stage
    int bpc;         // 32-row query blocks per copy: ceil(nq / 32) token blocks, or the group's queries
    int reps;        // copies of the blocks stacked in M (1, 2 or 4); they share a super-tile's columns
    int rows_alloc;  // query rows held per dimension chunk: 32 * bpc * reps
    uint32_t idesc;  // instruction descriptor, N field left 0 (set per super-tile)
    const uint8_t* pq_codes;    // kPQ: [n_tokens][16] uint8
    const float* pq_codebook;   // kPQ: [16][pq_k][8] fp32
    int pq_k;                   // kPQ: centroids per subspace (codes >= pq_k read zeros)
    long long budget;           // SM cycles a pipeline wait may last (<= 0: kWaitBudgetCycles)
    int fault;                  // diagnostics: kFaultHoldAccumulator, else 0
};

// Stands in for the row scale of a column past its document's end.
static __device__ const float kNanScale = __builtin_nanf("");

// Diagnostics (tms_debug_set): the MMA warp of CTA 0 never signals its
// first accumulator, so that CTA's epilogue wait runs out of budget and the
// timeout path -- flag, abort, drain, tensor-memory release -- runs.
constexpr int kFaultHoldAccumulator = TMS_FAULT_HOLD_ACCUMULATOR;

struct Layout {
    int q_off, qlo_off, stage_off, stage_stride, um_off, um_stride, fin_off, bias_off, deal_off, sc_off, cb_off, code_off, st_off, bar_off,
        misc_off, total;
};

// Per-query lists: super-tiles whose row maxima (up to 16 KB each) may wait for
// the finisher.  One leaves room for another chunk stage, and is enough where
// a super-tile takes three or more of them: 10 queries of 125 tokens x 2,948
// documents on the FP8 store at d = 768 took 467 us with two, and so two
// stages, 432 before there was a finisher, 381 with one.
constexpr int kMaxUmSlots = 2;
__host__ __device__ constexpr int um_slots(int nchunks) { return nchunks >= 3 ? 1 : kMaxUmSlots; }
// Finished documents waiting for their sum over query tokens, per epilogue warp
// (shared lists) or the finisher: kFinRows rows of 32 row maxima (one row per document and 32-row
// block), padded to 33 floats so that lane r reading row r walks distinct
// banks, then each row's (candidate, query) pair.  A group of four units ends
// at most four documents, so a group starts with at most kFinRows - 4 in use.
constexpr int kFinRows = 8;
constexpr int kFinWarpBytes = kFinRows * 33 * 4 + kFinRows * 8;

// Shared-memory carve-up; the same arithmetic runs on host and device.
// The query region comes first: the MMA reads 128 (x H) rows from each
// query chunk, and rows past rows_alloc fall on the following chunk or on
// the stage ring -- always inside the allocation, and they only feed
// accumulator rows that nothing reads.  A stage holds the full super-tile
// of str rows, so the document operand (N <= str) never reads past it.
// TF: the query region and every stage have a lo twin right after them.
// F8: per super-tile record slot, the row scale of every column.  Per-query
// lists: the sampled lengths (tms_deal.cuh).
// Streamed query (qslots = 0, qrows = 128 H): no resident query region;
// each chunk stage holds the str document rows, then the qrows query rows
// of the same dimension chunk.
__host__ __device__ inline Layout make_layout(int stages, int qslots, int nchunks, int rows_alloc, int str, int kind,
                                              int kacc, int blocks, bool sh, int qrows, int h, bool qt) {
    const bool f8 = kind == kE4M3;
    const int twin = kind == kTF32 ? 2 : 1;
    Layout L;
    L.q_off = 0;
    L.qlo_off = qslots * nchunks * rows_alloc * 128;
    L.stage_off = ((qt ? 1 : twin) * L.qlo_off + 1023) & ~1023;
    L.stage_stride = twin * (str + qrows) * 128;
    L.um_off = L.stage_off + stages * L.stage_stride;
    L.um_stride = sh ? 0 : (str / 8) * blocks * 128;  // [unit][32-row block][row] row maxima
    L.fin_off = L.um_off + um_slots(nchunks) * L.um_stride;
    L.bias_off = (L.fin_off + (sh ? epi_warps(h) : 1) * kFinWarpBytes + 127) & ~127;
    L.deal_off = L.bias_off + 256;
    L.sc_off = L.deal_off + (sh ? 0 : static_cast<int>(sizeof(deal::Shared)));
    L.cb_off = L.sc_off + (f8 ? st_ring(str) * str * 4 : 0);  // F8: [st_ring][str] column scales
    L.code_off = L.cb_off + (kind == kPQ ? kPqCbBytes : 0);                        // kPQ: fp16 codebook
    L.st_off = L.code_off + (kind == kPQ ? kCodeRing * str * kPqM : 0);  // kPQ: code-row ring
    L.bar_off = L.st_off + st_ring(str) * static_cast<int>(sizeof(StSlot));
    const int nbar = 3 * stages + 2 * kacc + 3 * qslots + 3 * st_ring(str) + 2 * kMaxUmSlots + 1 + kMmaWarps + 2 * kCodeRing;
    L.misc_off = L.bar_off + nbar * 8;
    L.total = L.misc_off + 16;
    return L;
}

// Candidate metadata for the planner: lane l of the warp holds the raw
// entry of candidate window position l.  Loads are only issued here; they
// are classified (meta_status) when the window becomes current, one window
// later, so the planner never waits on them.
struct Meta {
    int64_t off;
    int len;
    int id;
};

// The work items of one CTA, numbered k = 0, 1, ..., in the order in which
// each lane takes its own: k = lane, lane + 32, ...
// Per-query lists: one part of the flat list (tms_deal.cuh).  Score and top-k
// of 24 queries x 100 and 16 x 1,000 candidates, every query dealt to every
// CTA: 42 and 92 us (fp16), 38 and 84 (FP8), 82 and 235 (fp32); in parts 28 and
// 79, 27 and 64, 49 and 212.
// Shared lists: the groups are taken in rounds of `round_groups` (the last
// round `last_groups`); in a round the CTAs are dealt to its groups in turn
// and a group's candidates to its CTAs in turn, so CTAs of different groups
// read the same documents at about the same time: from HBM once per round,
// and from L2 for the rest (group after group over the whole list, every
// group read all of it from HBM).
template <bool SH>
struct Work;

template <>
struct Work<true> {
    int64_t n;              // items of this CTA
    int n1, q1, c1, j1;     // full rounds: items of one, group offset, first candidate, stride
    int64_t full;           // items of all full rounds
    int ql, cl, jl;         // last round: group, first candidate, stride

    __device__ __forceinline__ Work(const Args& a, const deal::Shared&) {
        const int b = blockIdx.x, grid = gridDim.x;
        auto count = [&](int c, int j) {
            return c < j && c < a.n_cand ? static_cast<int>((a.n_cand - c + j - 1) / j) : 0;
        };
        q1 = b % a.round_groups;
        c1 = b / a.round_groups;
        j1 = grid / a.round_groups;
        n1 = a.rounds > 1 ? count(c1, j1) : 0;
        full = static_cast<int64_t>(a.rounds - 1) * n1;
        ql = (a.rounds - 1) * a.round_groups + b % a.last_groups;
        cl = b / a.last_groups;
        jl = grid / a.last_groups;
        n = full + count(cl, jl);
    }
    // Item k < n: its group and its entry of the list.
    __device__ __forceinline__ void at(const Args& a, int64_t k, int* q, int* pos) const {
        if (k < full) {
            const int r = static_cast<int>(k / n1);
            *q = r * a.round_groups + q1;
            *pos = static_cast<int>(c1 + (k - static_cast<int64_t>(r) * n1) * j1);
        } else {
            *q = ql;
            *pos = static_cast<int>(cl + (k - full) * jl);
        }
    }
};

// Few members: they stay in the planner's registers beside its windows (with the
// list's pointers and the part held here too, short FP8 rows took 2% longer).
template <>
struct Work<false> {
    int64_t n;  // items of this CTA
    int lo;     // its first place in the flat list
    int q;      // this lane's query
    deal::Columns cols;
    float parts;  // CTAs per candidate; -1: of each list, in `dealt`
    const deal::Shared& dealt;

    __device__ __forceinline__ Work(const Args& a, const deal::Shared& sh) : dealt(sh) {
        parts = static_cast<float>(static_cast<int>(gridDim.x)) / static_cast<float>(static_cast<int>(a.n_flat));
        begin(a, deal::equal_part(static_cast<int>(a.n_flat)));
    }
    // The part by the lists' lengths, if it is another one.
    __device__ __forceinline__ bool recut(const Args& a) {
        if (!dealt.part.uneven) return false;
        if (a.n_queries <= deal::kGroups) parts = -1.f;
        begin(a, dealt.part);
        return true;
    }
    __device__ __forceinline__ void begin(const Args& a, deal::Part p) {
        lo = p.lo;
        n = p.hi - p.lo;
        // the first query that ends past lo, 32 candidates for it at a time
        const int lane = threadIdx.x & 31;
        int base = 0;
        for (int span = a.n_queries - 1; span > 0;) {
            const int step = (span + 31) / 32;
            const int last = min((lane + 1) * step, span) - 1;  // of this lane's piece
            const bool before = lane * step < span && __ldg(a.cand_offsets + base + last + 1) <= lo;
            const int pieces = __popc(__ballot_sync(0xffffffffu, before));
            base += min(pieces * step, span);
            span = min(step, span - min(pieces * step, span)) - 1;
        }
        enter(a, base);
    }
    __device__ __forceinline__ int bound(const Args& a, int i) const {
        const int64_t x = __ldg(a.cand_offsets + i);
        return static_cast<int>(x < 0 ? 0 : (x > a.n_flat ? a.n_flat : x));
    }
    __device__ __forceinline__ void enter(const Args& a, int query) {
        q = query;
        int c0 = 0, end = static_cast<int>(a.n_flat);  // one query: the first ids need not wait for its bounds
        if (a.n_queries > 1) c0 = bound(a, q), end = bound(a, q + 1);
        cols.enter(c0, end, parts < 0.f ? __int_as_float(dealt.sums[q]) : parts);
    }
    // Item k < n: its query and its flat index.
    __device__ __forceinline__ void at(const Args& a, int64_t k, int* query, int* pos) {
        const int p = lo + static_cast<int>(k);
        if (p >= cols.end && q < a.n_queries - 1) {
            int next = q + 1;
            while (next < a.n_queries - 1 && p >= bound(a, next + 1)) ++next;
            enter(a, next);
        }
        *query = q;
        *pos = p < cols.c0 || p >= cols.end ? p : cols.at(p);  // outside: not a valid list
    }
};

// The lists' lengths for the planner, by WARPS warps that have nothing to do yet
// (`warp` of them, the last one decides).  Out of line: passes of one list, which
// do not call it, fetch their instructions cold as well (1 x 10,000 and top-k
// 0.6 us longer with it inlined).
template <int WARPS>
__device__ __noinline__ void sample_lists(const int64_t* offsets, const int32_t* ids, const int32_t* lengths,
                                          int64_t n_docs, int n_queries, int total, deal::Shared* dealt, int warp) {
    const deal::Lists l{offsets, ids, lengths, n_docs, n_queries, total};
    deal::sample<8, 16>(l, dealt->sums, warp, WARPS);
    if (warp == WARPS - 1) {
        named_barrier_sync<2, 32 * WARPS>();
        deal::uneven_part(l, *dealt);
        __threadfence_block();
        named_barrier_arrive<1, 64>();  // with the planner
    } else {
        __threadfence_block();
        named_barrier_arrive<2, 32 * WARPS>();
    }
}

__device__ __forceinline__ Meta load_meta(const Args& a, int id) {
    Meta m;
    m.id = id;
    m.off = 0;
    m.len = 0;
    if (id >= 0 && id < a.n_docs) {
        m.off = __ldg(a.offsets + id);
        m.len = __ldg(a.lengths + id);
    }
    return m;
}

// 0 ok, 1 bad id, 2 bad row range.
__device__ __forceinline__ int meta_status(const Args& a, int id, int64_t off, int len) {
    if (id < 0 || id >= a.n_docs) return 1;
    return (len < 0 || off < 0 || off + len > a.n_tokens) ? 2 : 0;
}

// Every lane waits, and so observes the phase (and what it publishes)
// itself; the vote makes the outcome the warp's.  Returns false on timeout /
// abort.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          unsigned int* err, long long budget) {
    const bool ok = mbar_wait(bar, parity, abort_flag, err, budget);
    return __all_sync(0xffffffffu, ok) != 0;
}

// Drain wait: bounded, but ignores the abort flag (used to let in-flight
// asynchronous work land before the CTA exits).
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > kWaitBudgetCycles) break;
    }
}

// x with its 13 low mantissa bits cleared: the TF32 value a kind::tf32 MMA
// reads from an fp32 element.
__device__ __forceinline__ float tf32_trunc(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

// Maxima of the four units (8 columns each) of 32 accumulator columns.
__device__ __forceinline__ void unit_maxima(const float (&v)[32], float (&um)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
        um[k] = fmax3(fmax3(v[8 * k], v[8 * k + 1], v[8 * k + 2]), fmax3(v[8 * k + 3], v[8 * k + 4], v[8 * k + 5]),
                      fmaxf(v[8 * k + 6], v[8 * k + 7]));
}

// Max of the columns of unit K that count, with b[0..1] their row of the bias
// table (0, or -inf for the columns past the document's end).
template <int K>
__device__ __forceinline__ float unit_max_bias(const float (&v)[32], const float4* b) {
    const float4 x = b[0], y = b[1];
    return fmax3(fmax3(v[8 * K] + x.x, v[8 * K + 1] + x.y, v[8 * K + 2] + x.z),
                 fmax3(v[8 * K + 3] + x.w, v[8 * K + 4] + y.x, v[8 * K + 5] + y.y),
                 fmaxf(v[8 * K + 6] + y.z, v[8 * K + 7] + y.w));
}

// Maxima of the four units from unit u on, whose columns are in v, with the
// columns past a document's end dropped.
__device__ __forceinline__ void unit_maxima_counted(const float (&v)[32], float (&um)[4], uint32_t partial,
                                                    const uint8_t* valid, const float* bias) {
    unit_maxima(v, um);
    if (partial != 0u) {
        const float4* b = reinterpret_cast<const float4*>(bias);
        if (partial & 1u) um[0] = unit_max_bias<0>(v, b + 2 * valid[0]);
        if (partial & 2u) um[1] = unit_max_bias<1>(v, b + 2 * valid[1]);
        if (partial & 4u) um[2] = unit_max_bias<2>(v, b + 2 * valid[2]);
        if (partial & 8u) um[3] = unit_max_bias<3>(v, b + 2 * valid[3]);
    }
}

// Tensor maps of one launch.  doc[h] covers document rows with a box of
// 8 (h + 1) rows x one 128-byte chunk, so a tile of r rows is always ONE
// box per chunk (at most 7 rows of over-fetch).
struct Maps {
    CUtensorMap q;
    CUtensorMap doc[kBoxKinds];
};

// H: 128-row halves of the query tile (2 for a shared group of 8 queries).
// STR: rows per super-tile (MMA N at most), 256 or 128.  CTAS: CTAs per SM
// (1 or 2); the CTA holds KACC = acc_count(...) accumulators of STR
// tensor-memory columns; half h of super-tile t is accumulator use H t + h.
// SH (shared mode): the launch's queries all score one candidate list; a
// "query" of the pipeline is then a group of up to 4 H queries stacked in
// M, so each document tile is read once per group, and the epilogue
// writes one score per query of the group.
// F8: rows are E4M3 codes; similarities are scaled by the document row's
// scale before the max and by the query token's scale before the sum.
// QT (TF): the query in tensor memory, see kQueryCols.
template <int H, int STR, int CTAS, bool SH, int KIND, bool QT = false>
__global__ void __launch_bounds__(kernel_threads(KIND, H, SH), CTAS)
    dense_tc_kernel(const __grid_constant__ Maps maps, const Args a) {
    constexpr bool F8 = KIND == kE4M3;
    constexpr bool TF = KIND == kTF32;
    constexpr bool PQ = KIND == kPQ;
    constexpr int CE = chunk_elems(KIND);
    constexpr int STAGE_BYTES = STR * 128;
    constexpr int KACC = acc_count(STR, CTAS, QT);
    constexpr uint32_t TCOLS = KACC * STR + (QT ? kQueryCols : 0);
    constexpr int kEpiWarps = epi_warps(H);
    constexpr int kLoaderWarp = 1 + kMmaWarps;
    constexpr int kEpiWarp = kLoaderWarp + 1;  // the first of them
    static_assert(kEpiWarp % 4 == 0, "epilogue warp w reads the tensor-memory lanes of quarter w % 4");
    constexpr int kFinWarp = kEpiWarp + kEpiWarps;         // the first of them
    constexpr int kHelpers = help_warps(KIND);
    constexpr int kHelpWarp = kFinWarp + fin_warps(SH);    // TF / kPQ: the first splitter / decompressor
    constexpr int kStRing = st_ring(STR);
    static_assert(KACC >= 2 && TCOLS * CTAS <= 512, "tensor memory of one SM");

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int S = a.stages;
    const int QS = a.qslots;
    const int NCH = a.nchunks;
    const int qslot_bytes = NCH * a.rows_alloc * 128;
    const bool QSTREAM = QS == 0;  // the query rows come with every chunk stage
    const Layout L = make_layout(S, QS, NCH, a.rows_alloc, STR, KIND, KACC, a.bpc, SH, QSTREAM ? 128 * H : 0, H, QT);
    const int UMS = um_slots(NCH);
    const int SSTRIDE = L.stage_stride;  // bytes between stages (TF: hi, then lo)

    uint8_t* q_base = smem + L.q_off;
    uint8_t* qlo_base = smem + L.qlo_off;  // TF: the lo twin of the query region
    uint8_t* stage_base = smem + L.stage_off;
    uint8_t* um_base = smem + L.um_off;    // per-query lists: [UMS][unit][block][row] row maxima
    uint8_t* fin_base = smem + L.fin_off;  // finished-document rows
    float* bias = reinterpret_cast<float*>(smem + L.bias_off);  // [8][8]: entry [n][j] 0 for j < n, else -inf
    deal::Shared& dealt = *reinterpret_cast<deal::Shared*>(smem + L.deal_off);  // per-query lists: see tms_deal.cuh
    float* sc = reinterpret_cast<float*>(smem + L.sc_off);      // F8: [kStRing][STR] scale of each column
    StSlot* slots = reinterpret_cast<StSlot*>(smem + L.st_off);
    uint8_t* cb = smem + L.cb_off;           // kPQ: fp16 codebook, entry (code, m) at (code * 16 + m) * 16
    uint8_t* code_ring = smem + L.code_off;  // kPQ: [kCodeRing][STR rows][16] code bytes
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.bar_off);
    uint64_t* full = bars;
    uint64_t* empty = full + S;
    uint64_t* tfull = empty + S;              // [KACC] accumulator ready
    uint64_t* tempty = tfull + KACC;          // [KACC] accumulator read by every active epilogue warp
    uint64_t* qfull = tempty + KACC;
    uint64_t* qempty = qfull + QS;
    uint64_t* xfull = qempty + QS;          // [kStRing]
    uint64_t* xempty = xfull + kStRing;     // [kStRing]
    uint64_t* umfull = xempty + kStRing;    // [UMS] row maxima written
    uint64_t* umempty = umfull + kMaxUmSlots;         // [UMS] row maxima read
    uint64_t* scfull = umempty + kMaxUmSlots;          // F8: [kStRing] a record slot's column scales landed
    uint64_t* qready = scfull + kStRing;     // QT: the query is in tensor memory
    uint64_t* mdone = qready + 1;
    uint64_t* conv = mdone + kMmaWarps;   // TF: [S] stage split
    uint64_t* qconv = conv + S;   // TF: [QS] query tile split
    uint64_t* codefull = qconv + QS;            // kPQ: [kCodeRing] code rows landed
    uint64_t* codeempty = codefull + kCodeRing;  // kPQ: [kCodeRing] code rows consumed
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L.misc_off);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L.misc_off + 4);

    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);  // the same in every lane
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int i = 0; i < S; ++i) {
            mbar_init(&full[i], PQ ? kHelpers : 1);  // kPQ: every decompressor warp wrote its rows
            mbar_init(&empty[i], kMmaWarps);  // the MMAs that read it, and the other MMA warps passing it
        }
        for (int i = 0; i < KACC; ++i) {
            mbar_init(&tfull[i], 1);
            // the epilogue warps of a half whose row block belongs to a copy, and the
            // other MMA warps passing it
            mbar_init(&tempty[i], (H == 1 && a.reps * a.bpc < 4 ? a.reps * a.bpc : 4) + kMmaWarps - 1);
        }
        for (int i = 0; i < QS; ++i) {
            mbar_init(&qfull[i], 1);
            // the MMAs of every MMA warp, or (QT) the copies to tensor memory
            mbar_init(&qempty[i], QT ? (a.reps * a.bpc < 4 ? a.reps * a.bpc : 4) : kMmaWarps);
        }
        for (int i = 0; i < kStRing; ++i) {
            mbar_init(&xfull[i], 1);
            // loader, MMA, epilogue, finishers, splitters
            mbar_init(&xempty[i], 1 + kMmaWarps + kEpiWarps + fin_warps(SH) + ((TF || PQ) ? kHelpers : 0));
        }
        for (int i = 0; i < kMaxUmSlots; ++i) {
            mbar_init(&umfull[i], a.reps * a.bpc < 4 ? a.reps * a.bpc : 4);
            mbar_init(&umempty[i], 1);
        }
        for (int i = 0; i < kStRing; ++i) mbar_init(&scfull[i], 32);  // one cp.async arrival per loader lane
        mbar_init(qready, (a.reps * a.bpc < 4 ? a.reps * a.bpc : 4) + kMmaWarps);
        for (int i = 0; i < kMmaWarps; ++i) mbar_init(&mdone[i], 1);
        for (int i = 0; i < S; ++i) mbar_init(&conv[i], kHelpers);
        for (int i = 0; i < QS; ++i) mbar_init(&qconv[i], kHelpers);
        for (int i = 0; i < kCodeRing; ++i) {
            mbar_init(&codefull[i], 1);
            mbar_init(&codeempty[i], kHelpers);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == kLoaderWarp) {
        if (lane < kBoxKinds) prefetch_tensormap(&maps.doc[lane]);
    }
    if (warp == 0 && lane == 0) prefetch_tensormap(&maps.q);
    if (warp == 0) {
        bias[lane] = (lane & 7) < lane >> 3 ? 0.f : -INFINITY;
        bias[32 + lane] = (lane & 7) < 4 + (lane >> 3) ? 0.f : -INFINITY;
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, TCOLS);
        tmem_relinquish();
    }
    // Nothing above reads global memory: the previous kernel of the stream
    // may still be running until here.
    griddep_wait();
    griddep_launch_dependents();
    if constexpr (PQ) {
        // the codebook, rounded to fp16 (nearest even), for all 256 codes:
        // codes >= pq_k get zeros
        for (int e = threadIdx.x; e < 256 * kPqM; e += blockDim.x) {
            const int code = e / kPqM;
            const int m = e - code * kPqM;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (code < a.pq_k) {
                const float4* src =
                    reinterpret_cast<const float4*>(a.pq_codebook + (static_cast<int64_t>(m) * a.pq_k + code) * 8);
                const float4 x0 = __ldg(src), x1 = __ldg(src + 1);
                const __half2 h0 = __floats2half2_rn(x0.x, x0.y), h1 = __floats2half2_rn(x0.z, x0.w);
                const __half2 h2 = __floats2half2_rn(x1.x, x1.y), h3 = __floats2half2_rn(x1.z, x1.w);
                v = make_uint4(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1),
                               *reinterpret_cast<const uint32_t*>(&h2), *reinterpret_cast<const uint32_t*>(&h3));
            }
            *reinterpret_cast<uint4*>(cb + e * 16) = v;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *tmem_slot;
    if (warp == 0) {
        // ------------------------------------------------------- planner
        const uint64_t pol_keep = policy_evict_last();
        int tst = 0;   // super-tiles published
        int qi = 0, cur_q = -1;
        bool aborted = false;
        // The open super-tile, written into its record slot as it fills.
        int used = 0, nseg = 0, nfin = 0, st_q = 0;  // units, tiles, documents ended, query
        unsigned ends = 0, partial = 0;
        uint32_t shares = 0x80000000u >> (32 - STR / 8);  // last units of the shares
        if (a.reps >= 2) shares |= shares >> (STR / 16);
        if (a.reps >= 4) shares |= shares >> (STR / 32);

        // Publish the open super-tile: the record, and the query tile if the
        // query changed.
        auto close_st = [&]() -> bool {
            const int xs = tst % kStRing;
            if (lane == 0) {
                StHdr h;
                h.q = st_q;
                h.n = (8 * used + 15) & ~15;
                h.nseg = nseg;
                h.flags = 0;
                h.rows = 8 * used;
                h.ends = ends;
                h.partial = partial;
                h.values = (shares & (used == 32 ? 0xffffffffu : (1u << used) - 1u)) | ends;
                slots[xs].h = h;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&xfull[xs]);
            ++tst;
            used = nseg = nfin = 0;
            ends = partial = 0;
            // A new query's rows go to the next query slot.  The record is
            // published first: the MMA warps release the old slot only
            // once they see the new query.
            if (!QSTREAM && st_q != cur_q) {
                const int slot = qi % QS;
                if (!warp_wait(&qempty[slot], ((qi / QS) & 1) ^ 1, abort_flag, a.err, a.budget)) return false;
                if (lane == 0) {
                    mbar_arrive_expect_tx(&qfull[slot], static_cast<uint32_t>(qslot_bytes));
                    uint8_t* qdst = q_base + slot * qslot_bytes;
                    for (int kc = 0; kc < NCH; ++kc) {
                        uint8_t* cdst = qdst + kc * a.rows_alloc * 128;
                        for (int rp = 0; rp < (QT ? 1 : a.reps); ++rp)
                            tma_load_3d(cdst + rp * a.bpc * 32 * 128, &maps.q, kc * CE, 0, st_q * (SH ? a.group : 1),
                                        &qfull[slot], pol_keep);
                    }
                }
                ++qi;
                cur_q = st_q;
            }
            return true;
        };

        if (!SH && blockIdx.x == 0 && lane == 0 && __ldg(a.cand_offsets + a.n_queries) != a.n_cand)
            atomicOr(a.err, TMS_DEVERR_BAD_CSR);
        // three-window metadata pipeline: ids two windows ahead, offsets
        // and lengths one window ahead, the current window in registers.
        Work<SH> work(a, dealt);
        struct Item {
            int q, pos, id;  // query (group), entry of the list (per-query lists: flat index), document
        };
        auto item = [&](int64_t k) {
            Item x{0, 0, -1};
            if (k < work.n) {
                work.at(a, k, &x.q, &x.pos);
                x.id = __ldg(a.cand_ids + x.pos);
            }
            return x;
        };
        Item now, then, later;
        Meta cur, nxt;
        for (bool recut = !SH && a.sampled;; recut = false) {
            now = item(lane);
            cur = load_meta(a, now.id);
            then = item(32 + lane);
            nxt = load_meta(a, then.id);
            later = item(64 + lane);
            if (!recut) break;
            if constexpr (!SH) {
                named_barrier_sync<1, 64>();  // the samples' loads ran beside these
                if (!work.recut(a)) break;
            }
        }

        for (int64_t k0 = 0;; k0 += 32) {
            if (k0 >= work.n) break;
            // lane = one candidate of the window
            const bool valid = k0 + lane < work.n;
            const int ql = now.q, pos = now.pos;
            const int status = valid ? meta_status(a, cur.id, cur.off, cur.len) : 3;
            if (valid && (status != 0 || cur.len == 0)) {
                const float v = status != 0 ? __int_as_float(0x7fc00000) : -INFINITY;
                if (SH) {
                    for (int g = 0; g < a.group; ++g)
                        if (ql * a.group + g < a.n_queries)
                            a.out[static_cast<int64_t>(ql * a.group + g) * a.n_cand + pos] = v;
                } else {
                    a.out[pos] = v;
                }
                if (status != 0) atomicOr(a.err, status == 1 ? TMS_DEVERR_BAD_ID : TMS_DEVERR_BAD_RANGE);
            }
            // Pack the window's documents, in order, into super-tiles: lane =
            // document, [b, e) its units counted from the open super-tile's
            // start.  Tiles of at most kRows rows fill a super-tile to its
            // last unit: a document that does not fit is cut at the
            // super-tile's end and continues in the next one.  All documents
            // of one query are placed by one scan, and each super-tile they
            // reach costs a fixed number of warp steps, whatever it holds
            // (a loop over the documents, a few shuffles each, took ~1,500
            // cycles per super-tile and bounded every 128-byte-row launch).
            const int len = valid && status == 0 ? cur.len : 0;
            const int nu = static_cast<int>((static_cast<unsigned>(len) + 7u) >> 3);
            const bool huge = __any_sync(0xffffffffu, nu > (1 << 25));  // then one by one: their sum may not fit
            int incl = nu;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += x;
            }
            const int row = static_cast<int>(cur.off);
            constexpr int C = STR / 8;  // units of a super-tile
            unsigned docs = __ballot_sync(0xffffffffu, nu > 0);
            while (docs != 0u) {
                const int first = __ffs(docs) - 1;
                const int q = __shfl_sync(0xffffffffu, ql, first);
                unsigned run = __ballot_sync(0xffffffffu, ql == q) & docs;  // consecutive among the documents
                if (huge) run &= 0u - run;
                docs &= ~run;
                if (used > 0 && q != st_q && !close_st()) {
                    aborted = true;
                    break;
                }
                st_q = q;
                const int base = used - __shfl_sync(0xffffffffu, incl - nu, first);
                const bool in = (run >> lane) & 1u;
                int e = huge ? used + nu : base + incl, b = e - nu;
                int end = __shfl_sync(0xffffffffu, e, 31 - __clz(run));  // units from the open super-tile's start
                int done = 0;  // units of this lane's document in earlier super-tiles
                for (;;) {
                    const int xs = tst % kStRing;
                    if (used == 0 && !warp_wait(&xempty[xs], ((tst / kStRing) & 1) ^ 1, abort_flag, a.err, a.budget)) {
                        aborted = true;
                        break;
                    }
                    StSlot* x = &slots[xs];
                    const int lo = max(b, 0), hi = min(e, C);
                    const int n = in && hi > lo ? hi - lo : 0;  // units here: one tile, or two if more than kRows rows
                    const bool two = n > kRows / 8;
                    const bool last = n > 0 && e <= C;
                    const unsigned m1 = __ballot_sync(0xffffffffu, n > 0), m2 = __ballot_sync(0xffffffffu, two);
                    const unsigned ml = __ballot_sync(0xffffffffu, last);
                    const unsigned below = (1u << lane) - 1u;
                    if (n > 0) {
                        SegInfo* sg = x->seg + nseg + __popc(m1 & below) + __popc(m2 & below);
                        const int rows = min(8 * n, len - 8 * done);
                        sg->row0 = row + 8 * done;
                        sg->nu = static_cast<uint8_t>(two ? kRows / 8 : n);
                        sg->cu = static_cast<uint8_t>(lo);
                        sg->rows = static_cast<uint16_t>(min(rows, kRows));
                        if (two) {
                            sg[1].row0 = row + 8 * done + kRows;
                            sg[1].nu = static_cast<uint8_t>(n - kRows / 8);
                            sg[1].cu = static_cast<uint8_t>(lo + kRows / 8);
                            sg[1].rows = static_cast<uint16_t>(rows - kRows);
                        }
                        if (last) {
                            x->f[nfin + __popc(ml & below)] = pos;
                            x->valid[hi - 1] = static_cast<uint8_t>(len - 8 * (nu - 1));
                        }
                        done += n;
                    }
                    const unsigned bit = last ? 1u << (hi - 1) : 0u;
                    ends |= __reduce_or_sync(0xffffffffu, bit);
                    partial |= __reduce_or_sync(0xffffffffu, (len & 7) != 0 ? bit : 0u);
                    nseg += __popc(m1) + __popc(m2);
                    nfin += __popc(ml);
                    used = min(end, C);
                    if (used == C && !close_st()) {
                        aborted = true;
                        break;
                    }
                    if (end <= C) break;
                    b -= C;
                    e -= C;
                    end -= C;
                }
                if (aborted) break;
            }
            if (aborted) break;
            now = then;
            cur = nxt;
            then = later;
            nxt = load_meta(a, then.id);
            later = item(k0 + 96 + lane);
        }
        if (!aborted && used > 0 && !close_st()) aborted = true;
        if (!aborted) {
            const int xs = tst % kStRing;
            if (warp_wait(&xempty[xs], ((tst / kStRing) & 1) ^ 1, abort_flag, a.err, a.budget) && lane == 0) {
                StHdr h;
                h.q = 0;
                h.n = 0;
                h.nseg = 0;
                h.flags = kEnd;
                h.rows = 0;
                h.ends = 0;
                h.partial = 0;
                h.values = 0;
                slots[xs].h = h;
                mbar_arrive(&xfull[xs]);
            }
        }
        // Let every copy this warp issued land before the CTA can exit.
        if (lane == 0) {
            // every query slot whose load may still be in flight (QS of them)
            const int nqs = qi < QS ? qi : QS;
            for (int i = 1; i <= nqs; ++i) drain_wait(&qfull[(qi - i) % QS], ((qi - i) / QS) & 1);
        }
        __syncwarp();
    } else if (PQ && warp == kLoaderWarp) {
        // --------------------------------------------------- loader (kPQ)
        // Each super-tile's code rows (16 bytes per token, one bulk copy per
        // tile) go to a ring slot; the decompressors turn them into rows.
        int64_t issued = 0;
        for (int t = 0;; ++t) {
            const int xs = t % kStRing;
            if (!warp_wait(&xfull[xs], (t / kStRing) & 1, abort_flag, a.err, a.budget)) break;
            const StHdr h = slots[xs].h;
            if (h.flags & kEnd) break;
            const bool has = lane < h.nseg;
            int r = 0, row0 = 0, col = 0;
            if (has) {
                const SegInfo si = slots[xs].seg[lane];
                row0 = si.row0;
                col = 8 * si.cu;
                r = si.rows;
            }
            int bytes = r * kPqM;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) bytes += __shfl_xor_sync(0xffffffffu, bytes, o);
            __syncwarp();
            if (lane == 0) mbar_arrive(&xempty[xs]);
            const int cs = t % kCodeRing;
            if (!warp_wait(&codeempty[cs], ((t / kCodeRing) & 1) ^ 1, abort_flag, a.err, a.budget)) break;
            if (lane == 0) mbar_arrive_expect_tx(&codefull[cs], static_cast<uint32_t>(bytes));
            __syncwarp();
            if (has)
                bulk_load(code_ring + (cs * STR + col) * kPqM, a.pq_codes + static_cast<int64_t>(row0) * kPqM,
                          static_cast<uint32_t>(r * kPqM), &codefull[cs]);
            ++issued;
        }
        // Let every copy still in flight land before the CTA can exit.
        if (lane == 0) {
            const int64_t n = issued < kCodeRing ? issued : kCodeRing;
            for (int64_t i = 1; i <= n; ++i)
                drain_wait(&codefull[(issued - i) % kCodeRing], static_cast<uint32_t>(((issued - i) / kCodeRing) & 1));
        }
        __syncwarp();
    } else if (warp == kLoaderWarp) {
        // -------------------------------------------------------- loader
        const uint64_t pol_stream = policy_evict_first();
        const uint64_t pol_keep = policy_evict_last();
        int s = 0;
        uint32_t ph = 0;
        int64_t issued = 0;
        int sc_sts = 0;  // F8: super-tiles whose column scales were issued
        for (int t = 0;; ++t) {
            const int xs = t % kStRing;
            if (!warp_wait(&xfull[xs], (t / kStRing) & 1, abort_flag, a.err, a.budget)) break;
            const StHdr h = slots[xs].h;
            if (h.flags & kEnd) break;
            const bool has = lane < h.nseg;
            int n8 = 8, row0 = 0, col = 0, rend = 0;
            if (has) {
                const SegInfo si = slots[xs].seg[lane];
                n8 = 8 * si.nu;
                row0 = si.row0;
                col = 8 * si.cu;
                rend = col + si.rows;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&xempty[xs]);
            if (F8) {
                // Each tile's row scales to its columns of the record slot's
                // scale array (4-byte copies: any row alignment), completing
                // on scfull[xs]; the columns past a document's end get NaN,
                // which every max drops.  A lane finds the tile of its
                // column by counting the tile starts up to its unit.  The
                // array is free: the slot was republished only after every
                // epilogue warp had finished with its previous use.
                float* dst = sc + xs * STR;
                const unsigned starts = __reduce_or_sync(0xffffffffu, has ? 1u << (col >> 3) : 0u);
                const int shift = row0 - col;  // row of column 0, were the tile to reach it
#pragma unroll
                for (int c0 = 0; c0 < STR; c0 += 32) {
                    const int c = c0 + lane;
                    const int i = max(__popc(starts & (2u * (1u << (c >> 3)) - 1u)) - 1, 0);
                    const int r = __shfl_sync(0xffffffffu, shift, i) + c;
                    const bool ok = c < __shfl_sync(0xffffffffu, rend, i);
                    if (c < h.rows) cp_async4(dst + c, ok ? a.t_scales + r : &kNanScale);
                }
                cp_async_mbar_arrive(&scfull[xs]);
                ++sc_sts;
            }
            const CUtensorMap* dmap = &maps.doc[(n8 >> 3) - 1];
            bool ok = true;
            for (int kc = 0; kc < NCH; ++kc) {
                if (!warp_wait(&empty[s], ph ^ 1, abort_flag, a.err, a.budget)) {
                    ok = false;
                    break;
                }
                if (lane == 0) {
                    mbar_arrive_expect_tx(&full[s], static_cast<uint32_t>((h.rows + (QSTREAM ? a.rows_alloc : 0)) * 128));
                    if (QSTREAM) {
                        // the query (group) rows of this chunk, laid out as one
                        // chunk of the resident query region
                        uint8_t* qdst = stage_base + s * SSTRIDE + STR * 128;
                        for (int rp = 0; rp < a.reps; ++rp)
                            tma_load_3d(qdst + rp * a.bpc * 32 * 128, &maps.q, kc * CE, 0, h.q * (SH ? a.group : 1),
                                        &full[s], pol_keep);
                    }
                }
                __syncwarp();
                if (has) tma_load_2d(stage_base + s * SSTRIDE + col * 128, dmap, kc * CE, row0, &full[s], pol_stream);
                ++issued;
                if (++s == S) {
                    s = 0;
                    ph ^= 1;
                }
            }
            if (!ok) break;
        }
        // Let every copy still in flight land before the CTA can exit.
        if (F8) {
            cp_async_wait_all();
            __syncwarp();
            if (lane == 0) {
                const int n = sc_sts < kStRing ? sc_sts : kStRing;
                for (int i = 1; i <= n; ++i) drain_wait(&scfull[(sc_sts - i) % kStRing], ((sc_sts - i) / kStRing) & 1);
            }
        }
        if (lane == 0) {
            const int64_t n = issued < S ? issued : S;
            int ss = s;
            uint32_t pp = ph;
            for (int64_t i = 0; i < n; ++i) {
                if (--ss < 0) {
                    ss = S - 1;
                    pp ^= 1;
                }
                drain_wait(&full[ss], pp);
            }
        }
        __syncwarp();
    } else if (PQ && warp >= kHelpWarp) {
        // ------------------------------------------------- decompressors
        // Thread = (row, 16-byte unit) pairs of every chunk stage: the unit
        // u of row R in chunk kc is the fp16 centroid of subspace 8 kc + u
        // for that row's code, written at unit u ^ (R % 8) -- the 128-byte
        // swizzle TMA would have produced -- so the MMA reads decompressed
        // rows exactly as it reads loaded ones.  A quarter-warp covers one
        // row: eight subspaces, eight distinct codebook bank groups, one
        // 128-byte store.
        const int tid = (warp - kHelpWarp) * 32 + lane;
        constexpr int kDecThreads = 32 * kHelpers;
        int s = 0;
        uint32_t ph = 0;
        for (int t = 0;; ++t) {
            const int xs = t % kStRing;
            if (!warp_wait(&xfull[xs], (t / kStRing) & 1, abort_flag, a.err, a.budget)) break;
            const StHdr h = slots[xs].h;
            if (h.flags & kEnd) break;
            const int cs = t % kCodeRing;
            if (!warp_wait(&codefull[cs], (t / kCodeRing) & 1, abort_flag, a.err, a.budget)) break;
            const uint8_t* crow = code_ring + cs * STR * kPqM;
            bool ok = true;
            for (int kc = 0; kc < NCH; ++kc) {
                if (!warp_wait(&empty[s], ph ^ 1, abort_flag, a.err, a.budget)) {
                    ok = false;
                    break;
                }
                uint8_t* stg = stage_base + s * SSTRIDE;
                const int u = tid & 7;              // unit (subspace 8 kc + u) of every row this thread writes
                const int m = kc * 8 + u;
                // Rows tid / 8 + kRowStep j, eight per batch.  Every load of a
                // batch is unconditional (any code byte indexes inside the
                // codebook) and issued before the batch's stores, so the
                // dependent shared-memory loads of the eight rows overlap.
                constexpr int kBatch = 8;
                constexpr int kRowStep = kDecThreads / 8;
                for (int r0 = tid >> 3; r0 < h.rows; r0 += kRowStep * kBatch) {
                    uint4 v[kBatch];
#pragma unroll
                    for (int j = 0; j < kBatch; ++j) {
                        const int R = min(r0 + kRowStep * j, STR - 1);
                        const uint32_t code = crow[R * kPqM + m];
                        v[j] = *reinterpret_cast<const uint4*>(cb + (code * kPqM + m) * 16);
                    }
#pragma unroll
                    for (int j = 0; j < kBatch; ++j) {
                        const int R = r0 + kRowStep * j;
                        if (R < h.rows) *reinterpret_cast<uint4*>(stg + R * 128 + ((u ^ (R & 7)) << 4)) = v[j];
                    }
                }
                fence_proxy_async_smem();  // generic-proxy writes, read next by the tensor cores
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[s]);
                if (++s == S) {
                    s = 0;
                    ph ^= 1;
                }
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&codeempty[cs]);
                mbar_arrive(&xempty[xs]);
            }
        }
    } else if (TF && warp >= kHelpWarp) {
        // ------------------------------------------------------ splitters
        // Split each new query tile and every landed chunk stage: the MMA
        // reads an fp32 element as hi = tf32_trunc(x), so x stays in place
        // as its own hi part and lo = x - hi (exact, |lo| < 2^-10 |x|) goes
        // to the twin region; then publish the split to the MMA warps.
        // Elements are independent, so the 128-byte swizzle needs no
        // decoding: x and lo keep the same byte positions.
        const int tid = (warp - kHelpWarp) * 32 + lane;
        constexpr int kSplitThreads = 32 * kHelpers;
        auto split = [&](uint8_t* hi_p, uint8_t* lo_p, int bytes) {
            float4* hv = reinterpret_cast<float4*>(hi_p);
            float4* lv = reinterpret_cast<float4*>(lo_p);
#pragma unroll 1
            for (int v = tid; v < bytes / 16; v += 2 * kSplitThreads) {
                const bool two = v + kSplitThreads < bytes / 16;
                const float4 x = hv[v];
                const float4 y = hv[two ? v + kSplitThreads : v];
                lv[v] = make_float4(x.x - tf32_trunc(x.x), x.y - tf32_trunc(x.y), x.z - tf32_trunc(x.z),
                                    x.w - tf32_trunc(x.w));
                if (two)
                    lv[v + kSplitThreads] = make_float4(y.x - tf32_trunc(y.x), y.y - tf32_trunc(y.y),
                                                        y.z - tf32_trunc(y.z), y.w - tf32_trunc(y.w));
            }
            fence_proxy_async_smem();  // generic-proxy writes, read next by the tensor cores
            __syncwarp();
        };
        int s = 0;
        uint32_t ph = 0;
        int qi = 0, cur_q = -1;
        for (int t = 0;; ++t) {
            const int xs = t % kStRing;
            if (!warp_wait(&xfull[xs], (t / kStRing) & 1, abort_flag, a.err, a.budget)) break;
            const StHdr h = slots[xs].h;
            if (h.flags & kEnd) break;
            __syncwarp();
            if (lane == 0) mbar_arrive(&xempty[xs]);
            bool ok = true;
            if (!QT && h.q != cur_q) {
                const int slot = qi % QS;
                if (!warp_wait(&qfull[slot], (qi / QS) & 1, abort_flag, a.err, a.budget)) break;
                split(q_base + slot * qslot_bytes, qlo_base + slot * qslot_bytes, qslot_bytes);
                if (lane == 0) mbar_arrive(&qconv[slot]);
                ++qi;
                cur_q = h.q;
            }
            for (int kc = 0; kc < NCH; ++kc) {
                if (!warp_wait(&full[s], ph, abort_flag, a.err, a.budget)) {
                    ok = false;
                    break;
                }
                split(stage_base + s * SSTRIDE, stage_base + s * SSTRIDE + STAGE_BYTES, h.rows * 128);
                if (lane == 0) mbar_arrive(&conv[s]);
                if (++s == S) {
                    s = 0;
                    ph ^= 1;
                }
            }
            if (!ok) break;
        }
    } else if (warp <= kMmaWarps) {
        // ---------------------------------------------------------- MMA
        // The whole warp runs this role, so that its control flow and the
        // descriptors are uniform -- kept in uniform registers, where the
        // MMA takes them from; a loop that one lane runs alone moves each
        // of them there for every MMA -- and one elected lane issues.
        // Descriptors advance by adding the 16-byte-unit offset of each
        // K-step to a per-stage base.  Warp w issues super-tiles w,
        // w + kMmaWarps, ...; past the others it goes through the same waits,
        // and its arrivals are part of their stages' and accumulators' next
        // phases: a wait can tell a phase only from the one before it, so no
        // phase may complete before every MMA warp has seen its predecessor
        // (a warp that came 1 us late, on a cold instruction cache, waited
        // for a phase that needed its own next super-tile).
        const int mw = warp - 1;
        int s = 0;
        uint32_t ph = 0;
        int qi = 0, cur_q = -1, qslot = 0;
        bool any = false;
        const bool half_major = H == 2 && !QSTREAM && 2 * NCH <= S;
        const uint32_t stage_sa = smem_u32(stage_base);
        for (int t = 0;; ++t) {
            const int xs = t % kStRing;
            if (!warp_wait(&xfull[xs], (t / kStRing) & 1, abort_flag, a.err, a.budget)) break;
            const StHdr* x = &slots[xs].h;
            if (__any_sync(0xffffffffu, x->flags & kEnd)) break;
            const int xq = __reduce_max_sync(0xffffffffu, x->q);
            const int xn = __reduce_max_sync(0xffffffffu, x->n);
            if (elect_one()) mbar_arrive(&xempty[xs]);
            if (!QSTREAM && xq != cur_q) {
                if (QT) {
                    // this warp's arrival is part of the phase, so that it
                    // cannot complete before the last one was seen here
                    if (elect_one()) mbar_arrive(qready);
                    if (!warp_wait(qready, qi & 1, abort_flag, a.err, a.budget)) break;
                    tc_fence_after();
                } else {
                    if (cur_q >= 0 && elect_one()) mma_commit(&qempty[qslot]);
                    qslot = qi % QS;
                    if (!warp_wait(TF ? &qconv[qslot] : &qfull[qslot], (qi / QS) & 1, abort_flag, a.err, a.budget))
                        break;
                }
                ++qi;
                cur_q = xq;
            }
            bool ok = true;
            const uint32_t q_desc = desc_sw128(smem_u32(q_base) + static_cast<uint32_t>(qslot * qslot_bytes));
            const uint32_t qlo_desc = desc_sw128(smem_u32(qlo_base) + static_cast<uint32_t>(qslot * qslot_bytes));
            const uint32_t idesc = a.idesc | (static_cast<uint32_t>(xn >> 3) << 17);
            // K-steps of chunk kc, half hq (its operands in the current stage).
            auto issue = [&](int kc, int hq, bool last_use) {
                const int ab = (H * t + hq) % KACC;
                const uint32_t d_tmem = tbase + static_cast<uint32_t>(ab * STR);
                const uint32_t b_desc = desc_sw128(stage_sa + static_cast<uint32_t>(s * SSTRIDE));
                const uint32_t blo_desc = desc_sw128(stage_sa + static_cast<uint32_t>(s * SSTRIDE + STAGE_BYTES));
                const uint32_t qoff = QSTREAM ? 0u : static_cast<uint32_t>(((kc * a.rows_alloc + hq * 128) * 128) >> 4);
                const uint32_t a_desc =
                    QSTREAM ? desc_sw128(stage_sa + static_cast<uint32_t>(s * SSTRIDE + (STR + hq * 128) * 128))
                            : q_desc + qoff;
                const uint32_t q_tmem = tbase + static_cast<uint32_t>(KACC * STR + kc * 64);  // QT: hi, then lo
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const uint32_t accumulate = (kc > 0 || kk > 0) ? 1u : 0u;
                        if (QT) {  // the three products below, A in tensor memory
                            mma_tf32_ta(d_tmem, q_tmem + 8 * kk, b_desc + 2 * kk, idesc, accumulate);
                            mma_tf32_ta(d_tmem, q_tmem + 8 * kk, blo_desc + 2 * kk, idesc, 1u);
                            mma_tf32_ta(d_tmem, q_tmem + 32 + 8 * kk, b_desc + 2 * kk, idesc, 1u);
                        } else if (TF) {  // hi.hi + hi.lo + lo.hi
                            mma_tf32(d_tmem, a_desc + 2 * kk, b_desc + 2 * kk, idesc, accumulate);
                            mma_tf32(d_tmem, a_desc + 2 * kk, blo_desc + 2 * kk, idesc, 1u);
                            mma_tf32(d_tmem, qlo_desc + qoff + 2 * kk, b_desc + 2 * kk, idesc, 1u);
                        } else if (F8)
                            mma_f8(d_tmem, a_desc + 2 * kk, b_desc + 2 * kk, idesc, accumulate);
                        else
                            mma_f16(d_tmem, a_desc + 2 * kk, b_desc + 2 * kk, idesc, accumulate);
                    }
                    if (kc == NCH - 1 && (a.fault != kFaultHoldAccumulator || blockIdx.x != 0 || t != 0))
                        mma_commit(&tfull[ab]);
                    if (last_use) mma_commit(&empty[s]);
                }
            };
            auto acc_free = [&](int hq) {
                const int use = H * t + hq;
                const bool got = warp_wait(&tempty[use % KACC], ((use / KACC) & 1) ^ 1, abort_flag, a.err, a.budget);
                tc_fence_after();
                return got;
            };
            auto stage_full = [&]() {
                const bool got = warp_wait(TF ? &conv[s] : &full[s], ph, abort_flag, a.err, a.budget);
                tc_fence_after();
                return got;
            };
            auto advance = [&]() {
                if (++s == S) {
                    s = 0;
                    ph ^= 1;
                }
            };
            if (t % kMmaWarps != mw) {
#pragma unroll
                for (int hq = 0; hq < H; ++hq) {
                    ok = ok && acc_free(hq);
                    if (ok && elect_one()) mbar_arrive(&tempty[(H * t + hq) % KACC]);
                }
                for (int kc = 0; kc < NCH && ok; ++kc) {
                    ok = stage_full();
                    if (ok && elect_one()) mbar_arrive(&empty[s]);
                    advance();
                }
                if (!ok) break;
                continue;
            }
            any = true;
            if (H == 2 && STR == 256 && half_major) {
                // Half by half, where the ring holds the chunks of two
                // super-tiles: the first half's accumulator is ready, and
                // free again, half a super-tile earlier.
                const int s0 = s;
                const uint32_t ph0 = ph;
                ok = acc_free(0);
                for (int kc = 0; kc < NCH && ok; ++kc) {
                    ok = stage_full();
                    if (!ok) break;
                    issue(kc, 0, false);
                    advance();
                }
                if (!ok || !acc_free(H - 1)) break;
                s = s0;
                ph = ph0;
                for (int kc = 0; kc < NCH; ++kc) {
                    issue(kc, H - 1, true);
                    advance();
                }
            } else {
                for (int kc = 0; kc < NCH; ++kc) {
                    ok = stage_full();
                    if (!ok) break;
#pragma unroll
                    for (int hq = 0; hq < H; ++hq) {
                        if (kc == 0 && !acc_free(hq)) {
                            ok = false;
                            break;
                        }
                        issue(kc, hq, hq == H - 1);
                    }
                    if (!ok) break;
                    advance();
                }
                if (!ok) break;
            }
        }
        // Every MMA this warp issued must finish before TMEM is freed.
        if (any && elect_one()) {
            mma_commit(&mdone[mw]);
            drain_wait(&mdone[mw], 0);
        }
        __syncwarp();
    } else {
        // ---------------------------------------- epilogue and finisher
        // Epilogue: thread = query row 128 hh + 32 qd + lane of the warp's
        // half hh (TMEM lane 32 qd + lane).  A warp reduces its columns, in
        // groups of four units, to a running max that starts again after
        // each document's end.
        //   * Shared lists: a warp owns one query of the group and sees all
        //     columns, so the value at a document's end is the row's
        //     maximum; a document that goes on keeps it in a register.
        //   * Per-query lists: row block qd is copy qd / bpc of token block
        //     qd % bpc; the copies hold the same sums, so each takes its
        //     share of the columns and leaves its values -- at documents'
        //     ends and at its last unit -- to the finisher warp, which
        //     combines them.
        // What counts here is the number of instructions: the warps of the
        // SM issue 1.7 a cycle between them, whatever their number (walking
        // the documents in every warp took 500-600 instructions per 128
        // columns; values and finishers for shared lists too, 7,600 per
        // 256-row super-tile over all warps).
        //
        // Documents are finished in batches: their 32 row maxima (times the
        // query-token scales, F8; 0 past nq) go to the warp's rows in shared
        // memory, and when they are full lane r sums row r in token order
        // and stores the score -- the same fixed order for every document,
        // wherever it sits in a batch.
        if constexpr (!SH) {
            // nothing to do here yet: the lists' lengths for the planner
            if (a.sampled) {
                sample_lists<kEpiWarps + fin_warps(SH)>(a.cand_offsets, a.cand_ids, a.lengths, a.n_docs, a.n_queries,
                                                        static_cast<int>(a.n_flat), &dealt, warp - kEpiWarp);
            }
        }
        const bool finisher = !SH && warp >= kFinWarp;
        const int ew = finisher || !SH ? 0 : warp - kEpiWarp;
        float* fin_rows = reinterpret_cast<float*>(fin_base + ew * kFinWarpBytes);
        int* fin_ids = reinterpret_cast<int*>(fin_base + ew * kFinWarpBytes + kFinRows * 33 * 4);
        int nfin = 0;  // rows in use
        auto flush = [&]() {
            __syncwarp();
            if (lane < nfin) {
                float x[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) x[i] = fin_rows[lane * 33 + i];
                float sum = 0.f;
#pragma unroll
                for (int i = 0; i < 32; ++i) sum += x[i];
                const int f = fin_ids[2 * lane];
                const int qq = fin_ids[2 * lane + 1];  // shared lists: the row's query
                if (SH) {
                    if (qq < a.n_queries) a.out[static_cast<int64_t>(qq) * a.n_cand + f] = sum;
                } else {
                    a.out[f] = sum;
                }
            }
            __syncwarp();
            nfin = 0;
        };
        if (finisher) {
            // lane = row of a token block; m[b] is the running max of block
            // b's row over the current document's columns, carried from one
            // super-tile to the next when a document is cut at a
            // super-tile's end.  With several blocks per query (nq > 32)
            // each block is summed across the warp and the blocks are added
            // in order.
            float m[kMaxBlocks], qsc[kMaxBlocks];  // qsc, F8: the row's query-token scale
#pragma unroll
            for (int b = 0; b < kMaxBlocks; ++b) m[b] = -INFINITY, qsc[b] = 1.f;
            int qsc_q = -1;
            auto row_value = [&](int b) {
                return b * 32 + lane < a.nq ? (F8 ? m[b] * qsc[b] : m[b]) : 0.f;
            };
            for (int t = 0;; ++t) {
                const int xs = t % kStRing;
                if (!warp_wait(&xfull[xs], (t / kStRing) & 1, abort_flag, a.err, a.budget)) break;
                const StHdr xh = slots[xs].h;
                if (xh.flags & kEnd) break;
                if (F8 && xh.q != qsc_q) {
                    qsc_q = xh.q;
#pragma unroll
                    for (int b = 0; b < kMaxBlocks; ++b)
                        qsc[b] = b * 32 + lane < a.nq
                                     ? __ldg(a.q_scales + static_cast<int64_t>(xh.q) * a.nq + b * 32 + lane)
                                     : 0.f;
                }
                const int us = t % UMS;
                if (!warp_wait(&umfull[us], (t / UMS) & 1, abort_flag, a.err, a.budget)) break;
                const float* um = reinterpret_cast<const float*>(um_base + us * L.um_stride) + lane;
                uint32_t todo = xh.values;
                int e = 0;  // documents ended so far in this super-tile
#pragma unroll 1
                while (todo != 0u) {
                    const int u = __ffs(todo) - 1;
                    todo &= todo - 1u;
                    m[0] = fmaxf(m[0], um[u * a.bpc * 32]);
                    if (a.bpc > 1) {
#pragma unroll
                        for (int b = 1; b < kMaxBlocks; ++b)
                            if (b < a.bpc) m[b] = fmaxf(m[b], um[(u * a.bpc + b) * 32]);
                    }
                    if (((xh.ends >> u) & 1u) == 0u) continue;
                    const int f = slots[xs].f[e++];
                    if (a.bpc == 1) {
                        fin_rows[nfin * 33 + lane] = row_value(0);
                        if (lane == 0) fin_ids[2 * nfin] = f;
                        if (++nfin == kFinRows) flush();
                    } else {
                        // the blocks' sums over the warp, each as warp_sum
                        // has it, with the blocks dealt to quarters of the
                        // warp on the way: one at a time, four blocks'
                        // twenty shuffles in a row bounded short documents
                        // (8 x 10,000 of 16 tokens, 128 query tokens, d = 128:
                        // FP8 281 us, now 156; fp16 272, now 151)
                        const bool up16 = (lane & 16) != 0, up8 = (lane & 8) != 0;
                        const float x0 = row_value(0), x1 = row_value(1), x2 = row_value(2), x3 = row_value(3);
                        const float s0 = (up16 ? x2 : x0) + __shfl_xor_sync(0xffffffffu, up16 ? x0 : x2, 16);
                        const float s1 = (up16 ? x3 : x1) + __shfl_xor_sync(0xffffffffu, up16 ? x1 : x3, 16);
                        float sum = (up8 ? s1 : s0) + __shfl_xor_sync(0xffffffffu, up8 ? s0 : s1, 8);
#pragma unroll
                        for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                        float tot = sum;  // lane 0: block 0; block b in lanes 8 b on
#pragma unroll
                        for (int b = 1; b < kMaxBlocks; ++b) {
                            const float x = __shfl_sync(0xffffffffu, sum, 8 * b);
                            if (b < a.bpc) tot += x;
                            m[b] = -INFINITY;
                        }
                        if (lane == 0) a.out[f] = tot;
                    }
                    m[0] = -INFINITY;
                }
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&umempty[us]);
                    mbar_arrive(&xempty[xs]);
                }
            }
        } else {
            const int qd = warp & 3;
            const int hh = H == 2 ? (warp - kEpiWarp) >> 2 : 0;
            const int copy = SH ? 0 : qd / a.bpc;
            const int blk = 4 * hh + qd - copy * a.bpc;  // token block, or query of the group
            const bool active = SH ? blk < a.bpc : copy < a.reps;
            const int share = SH ? STR / 8 : STR / 8 / a.reps;  // units per copy, a multiple of 4
            const int ua = copy * share;                        // the warp's first
            // F8: columns are read in blocks, two columns of four rows per
            // thread and unit, so that a thread needs two row scales per unit
            // and not eight: broadcast to every lane, 32 scales per group
            // took more of the shared-memory pipe than the MMAs left (with
            // 256-column MMAs running, 42-61 cycles per group and SM against
            // 11 for the load and the maxima; measured).  m[i] is then the
            // running max of row lane / 4 + 8 (i % 2) + 16 (i / 2) over this
            // thread's columns, and `row` the row it speaks for once the four
            // threads of a row are combined.
            constexpr int MR = F8 ? 4 : 1;
            const int row = F8 ? (lane >> 2) + 8 * (lane & 1) + 16 * ((lane >> 1) & 1) : lane;
            float m[MR], qsc = 1.f;  // qsc, F8, shared lists: the row's query-token scale
#pragma unroll
            for (int i = 0; i < MR; ++i) m[i] = -INFINITY;
            // The row's running max; it starts again.
            auto take_max = [&]() -> float {
                float x = m[0];
                if constexpr (F8) {
                    const bool b0 = (lane & 1) != 0, b1 = (lane & 2) != 0;
                    const float y0 = fmaxf(b0 ? m[1] : m[0], __shfl_xor_sync(0xffffffffu, b0 ? m[0] : m[1], 1));
                    const float y1 = fmaxf(b0 ? m[3] : m[2], __shfl_xor_sync(0xffffffffu, b0 ? m[2] : m[3], 1));
                    x = fmaxf(b1 ? y1 : y0, __shfl_xor_sync(0xffffffffu, b1 ? y0 : y1, 2));
                }
#pragma unroll
                for (int i = 0; i < MR; ++i) m[i] = -INFINITY;
                return x;
            };
            int qsc_q = -1;
            int qi = 0, cur_q = -1;  // QT
            for (int t = 0;; ++t) {
                const int xs = t % kStRing;
                if (!warp_wait(&xfull[xs], (t / kStRing) & 1, abort_flag, a.err, a.budget)) break;
                const StHdr xh = slots[xs].h;
                if (xh.flags & kEnd) break;
                if (!active) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&xempty[xs]);
                    continue;
                }
                const int units = xh.rows >> 3;
                const int u1 = min(units, ua + share);
                const int us = t % UMS;
                float* um_out = reinterpret_cast<float*>(um_base + us * L.um_stride) + blk * 32 + row;
                const float* scol = sc + xs * STR;  // F8: scale of each column's document row
                const int use = H * t + hh;
                const int ab = use % KACC;
                const uint32_t tacc = tbase + (static_cast<uint32_t>(qd * 32) << 16) + static_cast<uint32_t>(ab * STR);
                const int qq = SH ? xh.q * a.group + blk : 0;
                if (SH && F8 && xh.q != qsc_q) {
                    qsc_q = xh.q;
                    qsc = row < a.nq && qq < a.n_queries
                              ? __ldg(a.q_scales + static_cast<int64_t>(qq) * a.nq + row)
                              : 0.f;
                }
                if (QT && xh.q != cur_q) {
                    // The new query's rows of this warp's block, split, from
                    // the swizzled tile to its lanes.  The MMAs on the old
                    // ones are done: this warp has seen all their commits.
                    const int slot = qi % QS;
                    if (!warp_wait(&qfull[slot], (qi / QS) & 1, abort_flag, a.err, a.budget)) break;
                    const int r = 32 * blk + lane;
#pragma unroll 1
                    for (int half = 0; half < 2 * NCH; ++half) {  // 16 elements
                        const uint4* src = reinterpret_cast<const uint4*>(
                            q_base + slot * qslot_bytes + ((half >> 1) * a.rows_alloc + r) * 128);
                        const uint32_t qaddr = tbase + (static_cast<uint32_t>(qd * 32) << 16) +
                                               static_cast<uint32_t>(KACC * STR + (half >> 1) * 64 + (half & 1) * 16);
                        uint32_t w[16];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint4 x = src[(4 * (half & 1) + i) ^ (r & 7)];
                            w[4 * i] = x.x, w[4 * i + 1] = x.y, w[4 * i + 2] = x.z, w[4 * i + 3] = x.w;
                        }
                        tmem_st16(qaddr, w);  // the MMA reads x as hi
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const float x = __uint_as_float(w[i]);
                            w[i] = __float_as_uint(x - tf32_trunc(x));
                        }
                        tmem_st16(qaddr + 32, w);
                    }
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(&qempty[slot]);
                        mbar_arrive(qready);
                    }
                    ++qi;
                    cur_q = xh.q;
                }
                if (!SH && !warp_wait(&umempty[us], ((t / UMS) & 1) ^ 1, abort_flag, a.err, a.budget)) break;
                if (F8 && !warp_wait(&scfull[xs], (t / kStRing) & 1, abort_flag, a.err, a.budget)) break;
                if (!warp_wait(&tfull[ab], (use / KACC) & 1, abort_flag, a.err, a.budget)) break;
                tc_fence_after();
                const int* ended = slots[xs].f;  // SH: the documents that end here
                // Unit u ends a document: its row maximum is x.
                auto end_doc = [&](int u, float x) {
                    if (SH) {
                        fin_rows[nfin * 33 + row] = row < a.nq ? (F8 ? x * qsc : x) : 0.f;
                        ++nfin;
                    } else {
                        um_out[u * a.bpc * 32] = x;
                    }
                };
#pragma unroll 1
                for (int u = ua; u < u1; u += 4) {  // a group of four units: 32 columns
                    const uint32_t eg = (xh.ends >> u) & 15u;
                    const uint32_t taddr = tacc + static_cast<uint32_t>(8 * u);
                    auto landed = [&]() {  // after the last load: hand the accumulator back
                        if (u + 4 >= u1) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&tempty[ab]);
                        }
                    };
                    auto list_ended = [&]() {
                        if (SH) {
                            const int n = __popc(eg);
                            if (lane < n) {
                                fin_ids[2 * (nfin + lane)] = ended[lane];
                                fin_ids[2 * (nfin + lane) + 1] = qq;
                            }
                            ended += n;
                        }
                    };
                    if constexpr (F8) {
                        uint32_t r[2][16];
                        tmem_ld_blocks(taddr, r);
                        landed();
                        const float2* scales = reinterpret_cast<const float2*>(scol + 8 * u) + (lane & 3);
                        float v[4][MR][2];  // [unit][row][column], scaled; columns past a document's end are NaN
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const float2 sc2 = scales[4 * k];
#pragma unroll
                            for (int i = 0; i < MR; ++i) {
                                v[k][i][0] = __uint_as_float(r[i >> 1][4 * k + 2 * (i & 1)]);
                                v[k][i][1] = __uint_as_float(r[i >> 1][4 * k + 2 * (i & 1) + 1]);
                                mul_f32x2(v[k][i][0], v[k][i][1], sc2.x, sc2.y);
                            }
                        }
                        if (eg == 0u) {
#pragma unroll
                            for (int i = 0; i < MR; ++i)
#pragma unroll
                                for (int k = 0; k < 4; ++k) m[i] = fmax3(m[i], v[k][i][0], v[k][i][1]);
                            continue;
                        }
                        list_ended();
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
#pragma unroll
                            for (int i = 0; i < MR; ++i) m[i] = fmax3(m[i], v[k][i][0], v[k][i][1]);
                            if ((eg >> k) & 1u) end_doc(u + k, take_max());
                        }
                    } else {
                        float v[32], um[4];
                        tmem_ld32(taddr, v);
                        landed();
                        unit_maxima_counted(v, um, (xh.partial >> u) & 15u, slots[xs].valid + u, bias);
                        if (eg == 0u) {
                            m[0] = fmax3(m[0], fmax3(um[0], um[1], um[2]), um[3]);
                            continue;
                        }
                        list_ended();
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            m[0] = fmaxf(m[0], um[k]);
                            if ((eg >> k) & 1u) end_doc(u + k, take_max());
                        }
                    }
                    if (SH && nfin > kFinRows - 4) flush();
                }
                if (ua >= u1) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[ab]);
                }
                // the share's last unit, unless a document (or the super-tile) ended before or there
                if (!SH && ua + share <= units && ((xh.ends >> (ua + share - 1)) & 1u) == 0u)
                    end_doc(ua + share - 1, take_max());
                // nothing goes on; m may hold columns past the super-tile's last unit
                if (!SH || ((xh.ends >> (units - 1)) & 1u) != 0u) {
#pragma unroll
                    for (int i = 0; i < MR; ++i) m[i] = -INFINITY;
                }
                __syncwarp();
                if (lane == 0) {
                    if (!SH) mbar_arrive(&umfull[us]);
                    mbar_arrive(&xempty[xs]);
                }
            }
        }
        if (nfin > 0) flush();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tbase, TCOLS);
    }
}

// A launch configuration -- the kernel's counterpart of the paper's tile
// shape (Section 6.9, Table tile_ablation): rows per super-tile (documents
// per MMA run) and CTAs per SM, copies of the query blocks stacked in M
// (query tokens per epilogue warp), at most `stages` chunk stages (0: as
// many as fit), `qslots` resident query-tile slots (0: whichever gives
// more stages), or (qstream) the query streamed with each chunk stage
// instead of held resident -- the paper's dimension tiling applied to the
// query tile too.
struct Config {
    int str;
    int ctas;
    int reps;
    int stages;
    int qslots;
    int qstream;
};

// Configurations chosen by the autotuner, per device and launch shape.
struct TuneKey {
    int device, kind, h, sh, nchunks, bpc;
    bool operator<(const TuneKey& o) const {
        const int x[6] = {device, kind, h, sh, nchunks, bpc};
        const int y[6] = {o.device, o.kind, o.h, o.sh, o.nchunks, o.bpc};
        for (int i = 0; i < 6; ++i)
            if (x[i] != y[i]) return x[i] < y[i];
        return false;
    }
};
inline std::mutex& tune_mutex() {
    static std::mutex m;
    return m;
}
inline std::map<TuneKey, Config>& tune_table() {
    static std::map<TuneKey, Config> t;
    return t;
}
// Shared candidate lists: the query group size the autotuner chose, per
// device, row type, dimension chunks and queries per launch (capped at 8).
inline std::map<TuneKey, int>& group_table() {
    static std::map<TuneKey, int> t;
    return t;
}
inline TuneKey group_key(int device, int kind, int nchunks, int n_queries) {
    return TuneKey{device, kind, 0, 1, nchunks, n_queries < 8 ? n_queries : 8};
}

// The configurations an instantiation has kernels for.
template <int H, bool SH, int KIND>
inline int config_shapes(Config* out) {
    if (H == 2 && KIND != kPQ) {
        out[0] = {256, 1, 0, 0, 0, 0};
        out[1] = {128, 1, 0, 0, 0, 0};
        return 2;
    }
    if (H == 2 || KIND == kTF32) {
        out[0] = {128, 1, 0, 0, 0, 0};
        return 1;
    }
    if (KIND == kPQ) {  // one query half
        out[0] = {256, 1, 0, 0, 0, 0};
        return 1;
    }
    out[0] = {256, 1, 0, 0, 0, 0};
    out[1] = {128, 1, 0, 0, 0, 0};
    out[2] = {128, 2, 0, 0, 0, 0};
    return 3;
}

// Plan shared memory, encode the tensor maps and launch dense_tc_kernel.
// Without a tuned or forced configuration: one CTA per SM with 256-row
// super-tiles (about two documents per MMA run); two CTAs with 128-row ones
// for short rows; one CTA with 128-row ones for eight queries of three or four
// chunks and split TF32; the query streamed where its tile leaves too few stages
// (plan_tc has the lines and the figures).  KIND selects the row type; kE4M3 ignores `dtype` (rows
// are E4M3 codes; t_scales in `a`).  The caller sets a.nchunks =
// ceil(d / chunk_elems(KIND)), and a.bpc: per-query ceil(nq / 32), shared mode
// the group size.  `force` (the autotuner's) overrides the choice;
// TMS_ERR_UNSUPPORTED when it does not fit.
// The resolved launch configuration: every field of Config set (qslots 0:
// the query is streamed).
struct Plan {
    int str, ctas, reps, stages, qslots;
    bool operator==(const Plan& o) const {
        return str == o.str && ctas == o.ctas && reps == o.reps && stages == o.stages && qslots == o.qslots;
    }
};

// Whether a launch keeps its query in tensor memory (see kQueryCols).
template <int KIND>
inline bool query_in_tmem(const Args& a) {
    return KIND == kTF32 && a.nchunks <= kQueryChunks;
}

// The configuration a launch of this instantiation takes: `force` if it
// fits (else TMS_ERR_UNSUPPORTED), else the autotuner's for this shape if
// one fits, else the default below.
template <int H, bool SH, int KIND>
tms_status plan_tc(const DeviceInfo& dev, const Args& a, const Config* force, Plan* out) {
    constexpr bool F8 = KIND == kE4M3;
    constexpr bool TF = KIND == kTF32;
    constexpr bool PQ = KIND == kPQ;
    (void)F8;
    // Shared-memory plan for (rows per super-tile, CTAs per SM, copies):
    // the query-slot count (2, else 1) that gives the most stages; the
    // plan fits with at least 4 chunk stages (2 with one CTA per SM).
    const int max_reps = SH ? 1 : (a.bpc == 3 ? 1 : 4 / a.bpc);
    const bool qt = query_in_tmem<KIND>(a);
    // Which shapes take split TF32 is a rule of its own, not what happens to
    // fit: the exact fp32 kernel takes the others, and the two differ in the
    // last bits.
    if (TF && (a.bpc * a.nchunks > 18 || a.nchunks > 17)) return TMS_ERR_UNSUPPORTED;
    auto fits = [&](int str, int ctas, int rp, int need, int& stages, int& qslots, int cap = 0, int want_qs = 0,
                    bool stream = false) {
        if (rp < 1 || rp > max_reps) return false;
        if (H == 2 && PQ && str != 128) return false;
        if (stream && (TF || PQ)) return false;  // their query tiles are split / decompressed in place
        const int limit = ctas == 2 ? dev.smem_per_sm / 2 - dev.smem_reserved - 1024
                                    : std::min(kSmemLimit, dev.max_smem_optin) - 1024;
        int best = -1;
        for (int qs = stream ? 0 : 2; qs >= (stream ? 0 : 1); --qs) {
            if (!stream && want_qs && qs != want_qs) continue;
            const Layout L0 = make_layout(0, qs, a.nchunks, 32 * a.bpc * (qt ? 1 : rp), str, KIND,
                                          acc_count(str, ctas, qt), a.bpc, SH, stream ? 128 * H : 0, H, qt);
            int sts = std::min(kMaxStages, (limit - L0.total) / (L0.stage_stride + 24));
            if (cap > 0 && sts > cap) sts = cap;
            if (sts > best) {
                best = sts;
                stages = sts;
                qslots = qs;
            }
        }
        return best >= std::max(need, ctas == 2 ? 4 : 2);
    };
    // default: as many copies as fit with 4 stages, else (one CTA) with 2 --
    // with 3 of 256 rows where the query can be streamed instead.  The streamed
    // tile leaves four of those, and two are too few to cover HBM: 4 x 8,000
    // documents, fp16, 128 query tokens, d = 448: 547 us resident, 473 streamed
    // (509 when the row maxima took no room and three stages were left); 96,
    // d = 640: 795 and 642 (691); 64, d = 960: 1,168 and 953 (1,081); FP8, 128,
    // d = 1,024: 627 and 511; shared by 4, fp16, d = 512: 251 and 197.  Three
    // resident stages are as good (96, d = 512: 511 and 512).
    auto plan = [&](int str, int ctas, int& stages, int& qslots, int& reps, int most = 4) {
        const int least = ctas == 2 ? 4 : (str == 256 && !TF && !PQ ? 3 : 2);
        for (int need : {4, least})
            for (int rp = std::min(max_reps, most); rp >= 1; rp /= 2)
                if (fits(str, ctas, rp, need, stages, qslots)) {
                    reps = rp;
                    return true;
                }
        return false;
    };
    int stages = 0, qslots = 1, reps = 0, str = 0, ctas = 0;
    Config tuned{0, 0, 0, 0, 0, 0};
    if (!force) {
        std::lock_guard<std::mutex> lk(tune_mutex());
        const auto it = tune_table().find(TuneKey{dev.ordinal, KIND, H, SH ? 1 : 0, a.nchunks, a.bpc});
        if (it != tune_table().end()) tuned = it->second;
    }
    const Config* want = force ? force : (tuned.ctas ? &tuned : nullptr);
    if (want) {
        if (fits(want->str, want->ctas, want->reps, 2, stages, qslots, want->stages, want->qslots, want->qstream != 0)) {
            str = want->str;
            ctas = want->ctas;
            reps = want->reps;
        } else if (force) {
            return TMS_ERR_UNSUPPORTED;
        }
    }
    if (ctas == 0) {
        if (PQ && H == 1) {
            if (plan(256, 1, stages, qslots, reps)) str = 256, ctas = 1;
        } else if (H == 2 && !PQ && a.nchunks <= 2 && fits(256, 1, 1, 3, stages, qslots)) {
            str = 256, ctas = 1, reps = 1;
        } else if (H == 2 && !PQ && a.nchunks >= 5) {
            // streamed, below: what the resident tile of eight queries leaves
            // is two or three 128-row stages (61 queries x 12,000 documents,
            // fp16, d = 320: 1,192 us resident, 1,117 streamed; 16 queries,
            // FP8, d = 640: 348 and 316)
        } else if (H == 2 || TF) {
            // eight queries of three or four chunks: 128-row super-tiles,
            // four accumulators and four stages or more (as above, fp16, d =
            // 192: 731 us against 772 with 256 rows and three stages; FP8, d
            // = 384: 203 and 229)
            if (plan(128, 1, stages, qslots, reps)) str = 128, ctas = 1;
        } else if (SH ? a.nchunks <= 2 : (a.nchunks == 1 || (a.nchunks == 2 && a.bpc >= 2))) {
            // Short rows (one chunk: FP8 at d <= 128, fp16 / bf16 at d <= 64;
            // two where each warp has all of a super-tile's columns or half
            // of them): a super-tile carries few bytes for its fixed pipeline
            // costs, so two CTAs per SM run two pipelines side by side.
            // Over 20,000 documents of 32..180 tokens, one CTA and two:
            // shared by 2..4 queries, d = 64, fp16 91 and 69 us, FP8 116 and
            // 87; d = 128, 94 and 85, 113 and 85.  Lists, 4 x 10,000, 64
            // query tokens: fp16 d = 64 152 and 121 us, d = 96 156 and 141,
            // d = 128 157 and 152; but with 32 tokens and d = 128 591 and 595
            // (8 x 20,000), and shared d = 256 167 and 168.  Two copies are
            // enough for one chunk of fp16: 359 us at 8 x 20,000, d = 64,
            // against 383 with four (FP8: 445 against 431).
            if (plan(128, 2, stages, qslots, reps, !SH && KIND == kF16 && a.nchunks == 1 ? 2 : 4)) str = 128, ctas = 2;
            else if (plan(256, 1, stages, qslots, reps)) str = 256, ctas = 1;
            else if (plan(128, 1, stages, qslots, reps)) str = 128, ctas = 1;
        } else if (plan(256, 1, stages, qslots, reps)) {
            str = 256, ctas = 1;
        }
    }
    if (ctas == 0 && !TF && !PQ) {
        // the resident query tile leaves no room: stream it with every chunk
        // stage (the copies a 128-row half needs, at least two stages)
        const int sh[2][2] = {{256, 1}, {128, 1}};
        for (int i = 0; i < 2 && ctas == 0; ++i)
            for (int rp = max_reps; rp >= 1 && ctas == 0; rp /= 2)
                if (fits(sh[i][0], sh[i][1], rp, 2, stages, qslots, 0, 0, true)) {
                    str = sh[i][0];
                    ctas = sh[i][1];
                    reps = rp;
                }
    }
    if (ctas == 0) return TMS_ERR_UNSUPPORTED;
    *out = Plan{str, ctas, reps, stages, qslots};
    return TMS_OK;
}

// Shared lists: the rounds in which `groups` groups share `grid` CTAs (see
// Work).  A round of g groups gives each floor(grid / g) CTAs, and takes as
// long as one of those works on its candidates, so few rounds (few passes over
// the documents) are weighed against CTAs left over: the fewest rounds that
// keep 97% of the CTAs busy, else those that keep most.  At most 16 groups at a
// time, so that they stay close to one another -- or as many as it takes to
// give every CTA a candidate, and of lists with fewer candidates than CTAs
// whole ones count, with as much again as one for the round itself.  In rounds
// of 16 groups whatever the list, 4,096 queries that share one document took
// 68 us on 16 CTAs (16 when the groups were not dealt in rounds), now 12.
inline void plan_rounds(int grid, int groups, int64_t n_cand, Args* a) {
    const bool few = n_cand < grid;
    const int most = static_cast<int>(std::max<int64_t>(16, grid / n_cand));
    double best = 0;
    for (int rounds = (groups + most - 1) / most; rounds <= groups; ++rounds) {
        const int full = (groups + rounds - 1) / rounds;
        if ((rounds - 1) * full >= groups) continue;
        const int last = groups - (rounds - 1) * full;
        if (grid / full == 0) continue;
        auto docs = [&](int g) {  // a CTA's documents in a round of g groups
            const int64_t ctas = grid / g;
            return few ? static_cast<double>((n_cand + ctas - 1) / ctas + 1) : static_cast<double>(n_cand) / ctas;
        };
        const double time = (rounds - 1) * docs(full) + docs(last);
        if (best == 0 || time < (few ? 0.95 : 1.0) * best) {
            best = time;
            a->rounds = rounds;
            a->round_groups = full;
            a->last_groups = last;
        }
        if (static_cast<double>(groups) * n_cand >= 0.97 * grid * best || (few && 2 * rounds >= best)) break;
    }
}

template <int H, bool SH, int KIND>
tms_status launch_tc(const DeviceInfo& dev, const void* queries, tms_dtype dtype, int n_queries, int nq, int d,
                     const void* doc_tokens, int64_t n_tokens, Args a, cudaStream_t stream,
                     const Config* force = nullptr) {
    constexpr bool F8 = KIND == kE4M3;
    constexpr bool TF = KIND == kTF32;
    constexpr bool PQ = KIND == kPQ;
    constexpr int CE = chunk_elems(KIND);
    Plan p;
    tms_status st = plan_tc<H, SH, KIND>(dev, a, force, &p);
    if (st != TMS_OK) return st;
    const int str = p.str, ctas = p.ctas, reps = p.reps, stages = p.stages, qslots = p.qslots;
    const CUtensorMapDataType tdt = F8   ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                                  : TF ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                  : dtype == TMS_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                      : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    const uint64_t row_bytes = static_cast<uint64_t>(d) * (F8 ? 1 : (TF ? 4 : 2));
    // With no document rows nothing is ever loaded through the document
    // maps; describe the query buffer so that they still encode.
    const void* dbase = n_tokens > 0 ? doc_tokens : queries;
    Maps maps;
    // one query's token blocks, or a group's queries of 32 rows each: rows past nq are zeros
    st = encode_tmap_3d(&maps.q, tdt, queries, d, static_cast<uint64_t>(nq), static_cast<uint64_t>(n_queries), row_bytes,
                        CE, static_cast<uint32_t>(SH ? 32 : 32 * a.bpc), static_cast<uint32_t>(SH ? a.bpc : 1));
    if (st != TMS_OK) return st;
    a.reps = reps;
    const bool qt = query_in_tmem<KIND>(a);
    a.rows_alloc = 32 * a.bpc * (qt ? 1 : reps);
    for (int h = 0; h < kBoxKinds; ++h) {
        if (PQ) {  // rows are decompressed in shared memory, never loaded by TMA
            maps.doc[h] = maps.q;
            continue;
        }
        st = encode_tmap_2d(&maps.doc[h], tdt, dbase, d, n_tokens, row_bytes, CE, static_cast<uint32_t>(8 * (h + 1)));
        if (st != TMS_OK) return st;
    }
    // format code 0 is f16 under kind::f16 and E4M3 under kind::f8f6f4; 2 is TF32
    a.idesc = make_idesc(128, 0, TF ? 2u : ((!F8 && dtype == TMS_BF16) ? 1u : 0u));
    a.stages = stages;
    a.qslots = qslots;
    const Layout L = make_layout(stages, qslots, a.nchunks, a.rows_alloc, str, KIND, acc_count(str, ctas, qt), a.bpc, SH,
                                 qslots == 0 ? 128 * H : 0, H, qt);
    const int smem = L.total + 1024;
    void (*kern)(const Maps, const Args);
    if constexpr (H == 2 && !PQ) {
        kern = str == 256 ? dense_tc_kernel<2, 256, 1, SH, KIND> : dense_tc_kernel<2, 128, 1, SH, KIND>;
    } else if constexpr (H == 2) {
        kern = dense_tc_kernel<2, 128, 1, SH, KIND>;
    } else if constexpr (PQ) {
        kern = dense_tc_kernel<1, 256, 1, true, kPQ>;  // H == 2 took the first branch
    } else if constexpr (TF) {
        kern = qt ? dense_tc_kernel<1, 128, 1, false, kTF32, true> : dense_tc_kernel<1, 128, 1, false, kTF32>;
    } else {
        kern = str == 256 ? dense_tc_kernel<1, 256, 1, SH, KIND>
                          : (ctas == 2 ? dense_tc_kernel<1, 128, 2, SH, KIND> : dense_tc_kernel<1, 128, 1, SH, KIND>);
    }
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
        return launch_status(cudaErrorInvalidValue);
    const int64_t grid = std::min<int64_t>(static_cast<int64_t>(dev.sm_count) * ctas, a.n_flat);
    a.sampled = !SH && a.n_queries > 1 && a.n_flat / grid >= kMinSampled;
    if (SH) plan_rounds(static_cast<int>(grid), static_cast<int>(a.n_flat / a.n_cand), a.n_cand, &a);
    return launch_status(launch_dependent(kern, dim3(static_cast<unsigned>(grid)), dim3(kernel_threads(KIND, H, SH)),
                                          static_cast<size_t>(smem), stream, maps, a));
}

// Autotuner: time every configuration this instantiation has kernels for
// that fits the launch -- super-tile shape x copies x query tile (resident
// in 1 or 2 slots, or streamed) x stage cap (all that fit / 4), skipping
// plans already timed -- with 3
// timed launches after one warm-up each (CUDA events on `stream`), remember
// the fastest for the launch shape, and report how many were timed and the
// best mean time per launch.  Each launch writes the scores, so the last
// (the chosen configuration, launched again) leaves them in place.
template <int H, bool SH, int KIND>
tms_status tune_tc(const DeviceInfo& dev, const void* queries, tms_dtype dtype, int n_queries, int nq, int d,
                   const void* doc_tokens, int64_t n_tokens, const Args& a, cudaStream_t stream, int* n_timed,
                   float* best_ms_out = nullptr, bool relaunch = true) {
    Config shapes[3];
    const int ns = config_shapes<H, SH, KIND>(shapes);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        (void)cudaGetLastError();
        return TMS_ERR_CUDA;
    }
    float best_ms = 0.f;
    Config best{0, 0, 0, 0, 0, 0};
    int timed = 0;
    tms_status st = TMS_OK;
    Plan seen[64];
    int nseen = 0;
    for (int i = 0; i < ns && st == TMS_OK; ++i) {
        for (int rp = 4; rp >= 1 && st == TMS_OK; rp /= 2) {
            for (int qs = 0; qs <= 2 && st == TMS_OK; ++qs) {  // 0: the query streamed
                for (int cap = 0; cap <= 4 && st == TMS_OK; cap += 4) {
                    const Config c{shapes[i].str, shapes[i].ctas, rp, cap, qs, qs == 0 ? 1 : 0};
                    Plan pl;
                    if (plan_tc<H, SH, KIND>(dev, a, &c, &pl) != TMS_OK) continue;
                    bool dup = false;
                    for (int j = 0; j < nseen; ++j) dup = dup || seen[j] == pl;
                    if (dup || nseen == 64) continue;
                    seen[nseen++] = pl;
                    tms_status r = launch_tc<H, SH, KIND>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens,
                                                          a, stream, &c);
                    if (r == TMS_ERR_UNSUPPORTED) continue;
                    if (r != TMS_OK) {
                        st = r;
                        break;
                    }
                    cudaEventRecord(e0, stream);
                    for (int k = 0; k < 3 && r == TMS_OK; ++k)
                        r = launch_tc<H, SH, KIND>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, a,
                                                   stream, &c);
                    cudaEventRecord(e1, stream);
                    float ms = 0.f;
                    if (r != TMS_OK || cudaEventSynchronize(e1) != cudaSuccess ||
                        cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
                        st = r != TMS_OK ? r : TMS_ERR_CUDA;
                        break;
                    }
                    ++timed;
                    if (best.ctas == 0 || ms < best_ms) {
                        best_ms = ms;
                        best = c;
                    }
                }
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    (void)cudaGetLastError();
    if (st != TMS_OK) return st;
    if (best.ctas == 0) return TMS_ERR_UNSUPPORTED;
    {
        std::lock_guard<std::mutex> lk(tune_mutex());
        tune_table()[TuneKey{dev.ordinal, KIND, H, SH ? 1 : 0, a.nchunks, a.bpc}] = best;
    }
    if (n_timed) *n_timed = timed;
    if (best_ms_out) *best_ms_out = best_ms / 3.f;
    // leave the scores of the chosen configuration in place
    return relaunch ? launch_tc<H, SH, KIND>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, a, stream,
                                             &best)
                    : TMS_OK;
}

// Shared candidate lists in groups of `group` queries stacked in M (group
// 8: two 128-row halves): launch, or (tune) time the configurations of
// that group size first.  a.nchunks and the list fields are set by the
// caller.
template <int KIND>
inline tms_status shared_group_launch(const DeviceInfo& dev, const void* queries, tms_dtype dtype, int n_queries, int nq,
                               int d, const void* doc_tokens, int64_t n_tokens, Args a, int group,
                               cudaStream_t stream, bool tune, int* n_timed, float* ms) {
    const int64_t n_groups = (n_queries + group - 1) / group;
    if (n_groups * a.n_cand >= (int64_t(1) << 31)) return TMS_ERR_UNSUPPORTED;
    a.n_flat = n_groups * a.n_cand;
    a.group = group;
    a.bpc = group;
    if (tune)
        return group == 8 ? tune_tc<2, true, KIND>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, a,
                                                    stream, n_timed, ms, false)
                          : tune_tc<1, true, KIND>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, a,
                                                    stream, n_timed, ms, false);
    return group == 8 ? launch_tc<2, true, KIND>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, a, stream)
                      : launch_tc<1, true, KIND>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, a, stream);
}

// Group sizes tried, largest first: up to 8 queries, no more than the
// launch has (rounded up to a power of two), at least 2.
inline int first_group(int n_queries) { return n_queries >= 5 ? 8 : (n_queries >= 3 ? 4 : 2); }

// Score (or tune, then score) shared candidate lists: the autotuner's group
// size for this shape if it has one and it fits, else the largest group
// whose stacked query tile fits shared memory.  Tuning times every group
// size's configurations and keeps the fastest group and configuration.
template <int KIND>
inline tms_status shared_run(const DeviceInfo& dev, const void* queries, tms_dtype dtype, int n_queries, int nq, int d,
                      const void* doc_tokens, int64_t n_tokens, const Args& a, cudaStream_t stream, bool tune,
                      int* n_configs) {
    const TuneKey gk = group_key(dev.ordinal, KIND, a.nchunks, n_queries);
    if (tune) {
        int best_group = 0, total = 0;
        float best_ms = 0.f;
        for (int group = first_group(n_queries); group >= 2; group /= 2) {
            int n = 0;
            float ms = 0.f;
            const tms_status st =
                shared_group_launch<KIND>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, a, group, stream,
                                          true, &n, &ms);
            if (st == TMS_ERR_UNSUPPORTED) continue;
            if (st != TMS_OK) return st;
            total += n;
            if (best_group == 0 || ms < best_ms) {
                best_group = group;
                best_ms = ms;
            }
        }
        if (best_group == 0) return TMS_ERR_UNSUPPORTED;
        {
            std::lock_guard<std::mutex> lk(tune_mutex());
            group_table()[gk] = best_group;
        }
        if (n_configs) *n_configs = total;
    }
    int tuned_group = 0;
    {
        std::lock_guard<std::mutex> lk(tune_mutex());
        const auto it = group_table().find(gk);
        if (it != group_table().end()) tuned_group = it->second;
    }
    if (tuned_group) {
        const tms_status st = shared_group_launch<KIND>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens,
                                                        a, tuned_group, stream, false, nullptr, nullptr);
        if (st != TMS_ERR_UNSUPPORTED) return st;
    }
    for (int group = first_group(n_queries); group >= 2; group /= 2) {
        const tms_status st = shared_group_launch<KIND>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, a,
                                                        group, stream, false, nullptr, nullptr);
        if (st != TMS_ERR_UNSUPPORTED) return st;
    }
    return TMS_ERR_UNSUPPORTED;
}

}  // namespace dense

}  // namespace tms
