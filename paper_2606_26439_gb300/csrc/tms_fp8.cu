// tms_fp8.cu -- the FP8 E4M3 token store: per-row quantization and MaxSim
// scoring of E4M3 codes with one fp32 scale per row.
//
// A stored row stands for the vector scale * decode(codes).  Scoring runs
// the tensor-core kernel of tms_dense_tc.cuh with tcgen05.mma kind::f8f6f4
// (E4M3 x E4M3, fp32 accumulation): the 128-byte chunks, swizzle and
// descriptors are byte-for-byte those of the fp16 path, a chunk just holds
// 128 elements, so each document row costs half the HBM bytes and half the
// MMAs.  The document row's scale multiplies its similarities before the
// max; the query token's scale multiplies the column max before the sum
// (both scales are >= 0, so this equals Eq. 1 on the dequantized vectors).
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "tms_dense_tc.cuh"

namespace tms {

namespace fp8 {

constexpr int kQuantWarps = 8;
constexpr int kQuantUnits = 4;  // 8-element units of a row per lane: d <= 1024 over 32 lanes

// Elements 8 u .. 8 u + 7 of x as fp32 (x 16-byte aligned).
template <int DT>
__device__ __forceinline__ void load8(const void* x, int64_t u, float (&v)[8]) {
    if (DT == TMS_F32) {
        const float4* p = static_cast<const float4*>(x) + 2 * u;
        const float4 a = __ldcs(p), b = __ldcs(p + 1);
        v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
        v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    } else {
        const uint4 w = __ldcs(static_cast<const uint4*>(x) + u);
        const uint32_t h[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 f = DT == TMS_F16 ? __half22float2(*reinterpret_cast<const __half2*>(&h[i]))
                                           : __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h[i]));
            v[2 * i] = f.x;
            v[2 * i + 1] = f.y;
        }
    }
}

// x / s rounded to nearest even, from r = RN(1 / s): Markstein's final
// division step (P. Markstein, "Computation of elementary functions on the
// IBM RISC System/6000 processor", 1990) -- with r the correctly rounded
// reciprocal and q within an ulp of x / s, q + r (x - q s) rounds to
// RN(x / s).  x r alone can be two ulps off, so the step runs twice: once
// to reach an ulp, once to round.  The residual is taken with its sign
// reversed so that x = -0 keeps its sign.  Exact while no residual
// underflows, which keeping s within kQuantMinScale .. kQuantMaxScale
// ensures for every quotient that does not round to code 0.
__device__ __forceinline__ float div_markstein(float x, float s, float r) {
    float q = x * r;
    q = fmaf(fmaf(q, s, -x), -r, q);
    return fmaf(fmaf(q, s, -x), -r, q);
}
constexpr float kQuantMinScale = 0x1p-60f, kQuantMaxScale = 0x1p60f;

// Two E4M3 codes (a in the low byte), nearest even, saturating.
__device__ __forceinline__ uint32_t encode2(float a, float b) {
    return __nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E4M3);
}

// Per row: amax (fp32), s = amax / 448, code = E4M3(x / s) rounded to
// nearest even with saturation, both quotients those of an IEEE fp32
// division.  LP lanes share a row (a warp takes 32 / LP rows at once), each
// with up to kQuantUnits of the row's 8-element units (l, l + LP, ...), all
// loaded before their arithmetic.
//
// Few lanes per row, so that a row's shuffles and its two reciprocals are
// spread over up to 32 elements per lane; for d > 64 every access still covers
// whole 32-byte sectors (narrower rows store 8-byte pieces of them, and 200 M
// fp16 elements take 105 us at d = 64, 132 at 32, 121 at 16, against 92 at 128;
// one warp per row took 820 to 3,155).  Bound by HBM once the arithmetic is small enough.  4 M
// fp16 rows of 128 (1.55 GB): one warp per row with 8-byte loads, an IEEE
// division and a one-element conversion per code took 1,042 us (ALU 48%
// busy, DRAM 18%); 16 lanes per row with one unit each 349 us (issue 61%
// busy); 245 us as it is (0.93 of the measured copy rate).
template <int DT, int LP>
__global__ void __launch_bounds__(kQuantWarps * 32)
    quantize_kernel(const void* __restrict__ x, int64_t rows, int d, uint8_t* __restrict__ codes,
                    float* __restrict__ scales) {
    const int lane = threadIdx.x & 31;
    const int l = lane & (LP - 1);
    const int units = d >> 3;  // per row
    griddep_wait();
    griddep_launch_dependents();
    const int64_t step = static_cast<int64_t>(gridDim.x) * kQuantWarps * (32 / LP);
    int64_t row = (static_cast<int64_t>(blockIdx.x) * kQuantWarps + (threadIdx.x >> 5)) * (32 / LP) + lane / LP;
    // rows of one warp step differ by lane: the warp leaves together
    for (; __any_sync(0xffffffffu, row < rows); row += step) {
        float v[kQuantUnits][8];
#pragma unroll
        for (int g = 0; g < kQuantUnits; ++g) {
            const int u = l + g * LP;
            if (row < rows && u < units) {
                load8<DT>(x, row * units + u, v[g]);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) v[g][i] = 0.f;
            }
        }
        float amax = 0.f;
#pragma unroll
        for (int g = 0; g < kQuantUnits; ++g)
#pragma unroll
            for (int i = 0; i < 8; i += 2) amax = fmax3(amax, fabsf(v[g][i]), fabsf(v[g][i + 1]));
#pragma unroll
        for (int o = LP / 2; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        const float s = amax >= kQuantMinScale && amax <= kQuantMaxScale ? div_markstein(amax, 448.f, 1.f / 448.f)
                                                                         : __fdiv_rn(amax, 448.f);
        if (row < rows) {
            if (l == 0) scales[row] = s;
            const bool plain = s >= kQuantMinScale && s <= kQuantMaxScale;
            const float r = __frcp_rn(s);
#pragma unroll
            for (int g = 0; g < kQuantUnits; ++g) {
                const int u = l + g * LP;
                if (u >= units) break;
                float y[8];
                if (plain) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) y[i] = div_markstein(v[g][i], s, r);
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) y[i] = s == 0.f ? 0.f : __fdiv_rn(v[g][i], s);
                }
                uint2 w;
                w.x = encode2(y[0], y[1]) | (encode2(y[2], y[3]) << 16);
                w.y = encode2(y[4], y[5]) | (encode2(y[6], y[7]) << 16);
                __stcs(reinterpret_cast<uint2*>(codes) + row * units + u, w);
            }
        }
    }
}

// The instantiation for d: a quarter as many lanes per row as it has
// 8-element units, rounded up to a power of two.
template <int DT>
cudaError_t launch_quantize(int sm_count, const void* x, int64_t rows, int d, uint8_t* codes, float* scales,
                            cudaStream_t stream) {
    auto go = [&](auto kernel, int lp) {
        const int64_t per_block = static_cast<int64_t>(kQuantWarps) * (32 / lp);
        const int64_t want = (rows + per_block - 1) / per_block;
        const unsigned grid = static_cast<unsigned>(std::min<int64_t>(want, int64_t(sm_count) * 8));
        return launch_dependent(kernel, dim3(grid), dim3(kQuantWarps * 32), 0, stream, x, rows, d, codes, scales);
    };
    const int units = d / 8;
    if (units <= 4) return go(quantize_kernel<DT, 1>, 1);
    if (units <= 8) return go(quantize_kernel<DT, 2>, 2);
    if (units <= 16) return go(quantize_kernel<DT, 4>, 4);
    if (units <= 32) return go(quantize_kernel<DT, 8>, 8);
    if (units <= 64) return go(quantize_kernel<DT, 16>, 16);
    return go(quantize_kernel<DT, 32>, 32);
}

inline bool aligned4(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }

// Host checks shared by both scoring entry points; fills the common Args.
tms_status prepare(const uint8_t* q_codes, const float* q_scales, int n_queries, int nq, int d,
                   const uint8_t* doc_codes, const float* doc_scales, int64_t n_tokens, const int64_t* doc_offsets,
                   const int32_t* doc_lengths, int64_t n_docs, const int32_t* cand_ids, int64_t n_cand,
                   float* out_scores, DeviceInfo* dev, dense::Args* a) {
    if (n_queries < 1 || n_queries > 4096 || nq < 1 || nq > 128 || d < 16 || d > 1024 || d % 16 != 0)
        return TMS_ERR_INVALID_ARG;
    if (n_tokens < 0 || n_tokens >= (int64_t(1) << 31) || n_docs < 0 || n_cand < 0 ||
        n_cand >= (int64_t(1) << 31))
        return TMS_ERR_INVALID_ARG;
    if (!q_codes || !q_scales || !aligned16(q_codes) || !aligned4(q_scales)) return TMS_ERR_INVALID_ARG;
    if (n_cand > 0 && (!cand_ids || !out_scores || !aligned16(cand_ids) || !aligned16(out_scores)))
        return TMS_ERR_INVALID_ARG;
    if (n_docs > 0 && (!doc_offsets || !doc_lengths || !aligned16(doc_offsets) || !aligned16(doc_lengths)))
        return TMS_ERR_INVALID_ARG;
    if (n_tokens > 0 && (!doc_codes || !doc_scales || !aligned16(doc_codes) || !aligned16(doc_scales)))
        return TMS_ERR_INVALID_ARG;
    tms_status st = current_device(dev);
    if (st != TMS_OK) return st;
    *a = dense::Args{};
    a->offsets = doc_offsets;
    a->lengths = doc_lengths;
    a->cand_ids = cand_ids;
    a->out = out_scores;
    a->q_scales = q_scales;
    a->t_scales = doc_scales;
    a->err = dev->err;
    a->budget = debug_wait_budget();
    a->fault = debug_fault();
    a->n_docs = n_docs;
    a->n_tokens = n_tokens;
    a->n_cand = n_cand;
    a->n_queries = n_queries;
    a->nq = nq;
    a->nchunks = (d + dense::chunk_elems(dense::kE4M3) - 1) / dense::chunk_elems(dense::kE4M3);
    return TMS_OK;
}

}  // namespace fp8

}  // namespace tms

extern "C" tms_status tms_quantize_e4m3(const void* x, tms_dtype dtype, int64_t rows, int d, uint8_t* codes,
                                        float* scales, cudaStream_t stream) {
    using namespace tms;
    if (dtype != TMS_F16 && dtype != TMS_BF16 && dtype != TMS_F32) return TMS_ERR_INVALID_ARG;
    if (rows < 0 || d < 16 || d > 1024 || d % 16 != 0) return TMS_ERR_INVALID_ARG;
    if (rows == 0) return TMS_OK;
    if (!x || !codes || !scales || !aligned16(x) || !aligned16(codes) || !fp8::aligned4(scales))
        return TMS_ERR_INVALID_ARG;
    DeviceInfo dev;
    tms_status st = current_device(&dev);
    if (st != TMS_OK) return st;
    switch (dtype) {
        case TMS_F16: return launch_status(fp8::launch_quantize<TMS_F16>(dev.sm_count, x, rows, d, codes, scales, stream));
        case TMS_BF16:
            return launch_status(fp8::launch_quantize<TMS_BF16>(dev.sm_count, x, rows, d, codes, scales, stream));
        default: return launch_status(fp8::launch_quantize<TMS_F32>(dev.sm_count, x, rows, d, codes, scales, stream));
    }
}

namespace tms {
namespace fp8 {

// tms_score_fp8 / tms_tune_fp8: the same checks, then launch (or tune).
tms_status score(const uint8_t* q_codes, const float* q_scales, int n_queries, int nq, int d,
                 const uint8_t* doc_codes, const float* doc_scales, int64_t n_tokens, const int64_t* doc_offsets,
                 const int32_t* doc_lengths, int64_t n_docs, const int32_t* cand_ids, const int64_t* cand_offsets,
                 int64_t n_cand, float* out_scores, cudaStream_t stream, bool tune, int* n_configs) {
    if (n_configs) *n_configs = 0;
    if (!cand_offsets || !aligned16(cand_offsets)) return TMS_ERR_INVALID_ARG;
    DeviceInfo dev;
    dense::Args a;
    tms_status st = prepare(q_codes, q_scales, n_queries, nq, d, doc_codes, doc_scales, n_tokens, doc_offsets,
                            doc_lengths, n_docs, cand_ids, n_cand, out_scores, &dev, &a);
    if (st != TMS_OK || n_cand == 0) return st;
    a.cand_offsets = cand_offsets;
    a.n_flat = n_cand;
    a.group = 0;
    a.bpc = (nq + 31) / 32;
    if (tune)
        return dense::tune_tc<1, false, dense::kE4M3>(dev, q_codes, TMS_F16, n_queries, nq, d, doc_codes, n_tokens, a,
                                                      stream, n_configs);
    return dense::launch_tc<1, false, dense::kE4M3>(dev, q_codes, TMS_F16, n_queries, nq, d, doc_codes, n_tokens, a,
                                                    stream);
}

// tms_score_fp8_shared / tms_tune_fp8_shared.
tms_status score_shared(const uint8_t* q_codes, const float* q_scales, int n_queries, int nq, int d,
                        const uint8_t* doc_codes, const float* doc_scales, int64_t n_tokens,
                        const int64_t* doc_offsets, const int32_t* doc_lengths, int64_t n_docs,
                        const int32_t* cand_ids, int64_t n_cand, float* out_scores, cudaStream_t stream, bool tune,
                        int* n_configs) {
    if (n_configs) *n_configs = 0;
    DeviceInfo dev;
    dense::Args a;
    tms_status st = prepare(q_codes, q_scales, n_queries, nq, d, doc_codes, doc_scales, n_tokens, doc_offsets,
                            doc_lengths, n_docs, cand_ids, n_cand, out_scores, &dev, &a);
    if (st != TMS_OK) return st;
    if (nq > 32) return TMS_ERR_UNSUPPORTED;
    if (n_cand == 0) return TMS_OK;
    a.cand_offsets = nullptr;
    return dense::shared_run<dense::kE4M3>(dev, q_codes, TMS_F16, n_queries, nq, d, doc_codes, n_tokens, a, stream,
                                           tune, n_configs);
}

}  // namespace fp8
}  // namespace tms

extern "C" tms_status tms_score_fp8(const uint8_t* q_codes, const float* q_scales, int n_queries, int nq, int d,
                                    const uint8_t* doc_codes, const float* doc_scales, int64_t n_tokens,
                                    const int64_t* doc_offsets, const int32_t* doc_lengths, int64_t n_docs,
                                    const int32_t* cand_ids, const int64_t* cand_offsets, int64_t n_cand,
                                    float* out_scores, cudaStream_t stream) {
    return tms::fp8::score(q_codes, q_scales, n_queries, nq, d, doc_codes, doc_scales, n_tokens, doc_offsets,
                           doc_lengths, n_docs, cand_ids, cand_offsets, n_cand, out_scores, stream, false, nullptr);
}

extern "C" tms_status tms_tune_fp8(const uint8_t* q_codes, const float* q_scales, int n_queries, int nq, int d,
                                   const uint8_t* doc_codes, const float* doc_scales, int64_t n_tokens,
                                   const int64_t* doc_offsets, const int32_t* doc_lengths, int64_t n_docs,
                                   const int32_t* cand_ids, const int64_t* cand_offsets, int64_t n_cand,
                                   float* out_scores, cudaStream_t stream, int* n_configs) {
    return tms::fp8::score(q_codes, q_scales, n_queries, nq, d, doc_codes, doc_scales, n_tokens, doc_offsets,
                           doc_lengths, n_docs, cand_ids, cand_offsets, n_cand, out_scores, stream, true, n_configs);
}

extern "C" tms_status tms_score_fp8_shared(const uint8_t* q_codes, const float* q_scales, int n_queries, int nq,
                                           int d, const uint8_t* doc_codes, const float* doc_scales,
                                           int64_t n_tokens, const int64_t* doc_offsets, const int32_t* doc_lengths,
                                           int64_t n_docs, const int32_t* cand_ids, int64_t n_cand,
                                           float* out_scores, cudaStream_t stream) {
    return tms::fp8::score_shared(q_codes, q_scales, n_queries, nq, d, doc_codes, doc_scales, n_tokens, doc_offsets,
                                  doc_lengths, n_docs, cand_ids, n_cand, out_scores, stream, false, nullptr);
}

extern "C" tms_status tms_tune_fp8_shared(const uint8_t* q_codes, const float* q_scales, int n_queries, int nq,
                                          int d, const uint8_t* doc_codes, const float* doc_scales,
                                          int64_t n_tokens, const int64_t* doc_offsets, const int32_t* doc_lengths,
                                          int64_t n_docs, const int32_t* cand_ids, int64_t n_cand,
                                          float* out_scores, cudaStream_t stream, int* n_configs) {
    return tms::fp8::score_shared(q_codes, q_scales, n_queries, nq, d, doc_codes, doc_scales, n_tokens, doc_offsets,
                                  doc_lengths, n_docs, cand_ids, n_cand, out_scores, stream, true, n_configs);
}
