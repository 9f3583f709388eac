// tms_dense.cu -- dense MaxSim entry points for fp16 / bf16 / fp32 rows.
//
// fp16 / bf16 run the tensor-core kernel of tms_dense_tc.cuh; fp32 too (split
// TF32) for up to 18 pairs of a 32-token query block and a 32-element chunk and
// up to 17 chunks, else an exact-fp32 CUDA-core kernel.
#include "tms_dense_tc.cuh"

namespace tms {

namespace dense {

// ------------------------------------------------------------------ fp32

constexpr int kF32Warps = 16;
constexpr int kF32Step = 8;  // dimensions per step: a 32-byte sector of a document row (d is a multiple of 8)

// Exact-fp32 MaxSim: one warp per candidate and block of 32 query tokens, the
// block's rows in shared memory with the dimension outermost ([d][32]).  Lane
// (tg, rg) = (lane / 8, lane % 8) holds the dot products of tokens 8 tg .. 8
// tg + 7 with four document rows, one fused multiply-add per dimension in
// ascending order, before the max.
//
// Bound by the FP32 pipes and the L1 return path together: a step's eight
// 16-byte loads of document rows (the next step's are in flight meanwhile) and
// sixteen of query tokens feed 256 multiply-adds per lane.  With one token per
// lane every 16 bytes loaded fed four: 8 queries x 15,650 documents of 1 to 64
// tokens, d = 768, took 52,400 us, now 14,800 (a quarter of the FP32 rate).
__global__ void __launch_bounds__(kF32Warps * 32, 1)
    dense_f32_kernel(const float* __restrict__ queries, const float* __restrict__ tokens, const Args a, int d) {
    extern __shared__ float qs[];  // [d][32]
    griddep_wait();
    griddep_launch_dependents();
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int tg = lane >> 3, rg = lane & 7;
    if (blockIdx.x == 0 && threadIdx.x == 0 && __ldg(a.cand_offsets + a.n_queries) != a.n_cand)
        atomicOr(a.err, TMS_DEVERR_BAD_CSR);
    for (int q = 0; q < a.n_queries; ++q) {
        int64_t c0 = __ldg(a.cand_offsets + q), c1 = __ldg(a.cand_offsets + q + 1);
        c0 = c0 < 0 ? 0 : (c0 > a.n_cand ? a.n_cand : c0);
        c1 = c1 < c0 ? c0 : (c1 > a.n_cand ? a.n_cand : c1);
        if (c0 + static_cast<int64_t>(blockIdx.x) * kF32Warps >= c1) continue;  // none for this CTA
        for (int ib = 0; ib < a.nq; ib += 32) {
            __syncthreads();
            for (int t = 4 * warp; t < d; t += 4 * kF32Warps) {  // lane = token
                const float4 x = ib + lane < a.nq
                                     ? __ldg(reinterpret_cast<const float4*>(
                                           queries + (static_cast<int64_t>(q) * a.nq + ib + lane) * d + t))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
                qs[t * 32 + lane] = x.x;
                qs[(t + 1) * 32 + lane] = x.y;
                qs[(t + 2) * 32 + lane] = x.z;
                qs[(t + 3) * 32 + lane] = x.w;
            }
            __syncthreads();
            for (int64_t c = c0 + static_cast<int64_t>(blockIdx.x) * kF32Warps + warp; c < c1;
                 c += static_cast<int64_t>(gridDim.x) * kF32Warps) {
                const int id = __ldg(a.cand_ids + c);
                int64_t off = 0;
                int len = 0;
                int status = 0;
                if (id < 0 || id >= a.n_docs) {
                    status = 1;
                } else {
                    off = __ldg(a.offsets + id);
                    len = __ldg(a.lengths + id);
                    if (len < 0 || off < 0 || off + len > a.n_tokens) status = 2;
                }
                if (status != 0 || len == 0) {
                    if (ib == 0 && lane == 0) {
                        if (status) {
                            a.out[c] = __int_as_float(0x7fc00000);
                            atomicOr(a.err, status == 1 ? TMS_DEVERR_BAD_ID : TMS_DEVERR_BAD_RANGE);
                        } else {
                            a.out[c] = -INFINITY;
                        }
                    }
                    continue;
                }
                float best[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) best[i] = -INFINITY;
                for (int j0 = 0; j0 < len; j0 += 32) {
                    // rows past the end repeat the last one: a max does not change
                    const float4* xr[4];
                    float4 x[4][2];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        xr[r] = reinterpret_cast<const float4*>(tokens + (off + min(j0 + 4 * rg + r, len - 1)) * d);
                        x[r][0] = __ldg(xr[r]);
                        x[r][1] = __ldg(xr[r] + 1);
                    }
                    float acc[4][8];
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int i = 0; i < 8; ++i) acc[r][i] = 0.f;
#pragma unroll 1
                    for (int t = 0; t < d; t += kF32Step) {
                        float4 n[4][2];
                        const int tn = t + kF32Step < d ? (t + kF32Step) / 4 : 0;  // the last step reloads the first
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            n[r][0] = __ldg(xr[r] + tn);
                            n[r][1] = __ldg(xr[r] + tn + 1);
                        }
#pragma unroll
                        for (int u = 0; u < kF32Step; ++u) {
                            const float4* qp = reinterpret_cast<const float4*>(qs + (t + u) * 32 + 8 * tg);
                            const float4 qa = qp[0], qb = qp[1];
                            const float qv[8] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w};
#pragma unroll
                            for (int r = 0; r < 4; ++r) {
                                const float4 y = x[r][u >> 2];
                                const float xv = (u & 3) == 0 ? y.x : (u & 3) == 1 ? y.y : (u & 3) == 2 ? y.z : y.w;
#pragma unroll
                                for (int i = 0; i < 8; ++i) acc[r][i] = fmaf(qv[i], xv, acc[r][i]);
                            }
                        }
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            x[r][0] = n[r][0];
                            x[r][1] = n[r][1];
                        }
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        best[i] = fmaxf(best[i], fmaxf(fmaxf(acc[0][i], acc[1][i]), fmaxf(acc[2][i], acc[3][i])));
                }
                // max over the eight row groups, halving the tokens each step:
                // lane 8 tg + rg ends with token 8 tg + rg
                float b4[4], b2[2];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const bool up = (rg & 4) != 0;
                    b4[i] = fmaxf(up ? best[4 + i] : best[i],
                                  __shfl_xor_sync(0xffffffffu, up ? best[i] : best[4 + i], 4));
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const bool up = (rg & 2) != 0;
                    b2[i] = fmaxf(up ? b4[2 + i] : b4[i], __shfl_xor_sync(0xffffffffu, up ? b4[i] : b4[2 + i], 2));
                }
                const bool up = (rg & 1) != 0;
                const float b1 = fmaxf(up ? b2[1] : b2[0], __shfl_xor_sync(0xffffffffu, up ? b2[0] : b2[1], 1));
                const float v = warp_sum(ib + lane < a.nq ? b1 : 0.f);
                if (lane == 0) a.out[c] = (ib == 0) ? v : a.out[c] + v;
            }
        }
    }
}

}  // namespace dense

}  // namespace tms

namespace tms {
namespace {

// tms_score_dense, or (tune) tms_tune_dense: the same checks and launch,
// the tensor-core configurations timed first.
tms_status score_dense(const void* queries, tms_dtype dtype, int n_queries, int nq, int d, const void* doc_tokens,
                       int64_t n_tokens, const int64_t* doc_offsets, const int32_t* doc_lengths, int64_t n_docs,
                       const int32_t* cand_ids, const int64_t* cand_offsets, int64_t n_cand, float* out_scores,
                       cudaStream_t stream, bool tune, int* n_timed) {
    if (n_timed) *n_timed = 0;
    if (dtype != TMS_F16 && dtype != TMS_BF16 && dtype != TMS_F32) return TMS_ERR_INVALID_ARG;
    if (n_queries < 1 || n_queries > 4096 || nq < 1 || nq > 128 || d < 8 || d > 1024 || d % 8 != 0)
        return TMS_ERR_INVALID_ARG;
    if (n_tokens < 0 || n_tokens >= (int64_t(1) << 31) || n_docs < 0 || n_cand < 0 ||
        n_cand >= (int64_t(1) << 31))
        return TMS_ERR_INVALID_ARG;
    if (!queries || !cand_offsets || !aligned16(queries) || !aligned16(cand_offsets)) return TMS_ERR_INVALID_ARG;
    if (n_cand > 0 && (!cand_ids || !out_scores || !aligned16(cand_ids) || !aligned16(out_scores)))
        return TMS_ERR_INVALID_ARG;
    if (n_docs > 0 && (!doc_offsets || !doc_lengths || !aligned16(doc_offsets) || !aligned16(doc_lengths)))
        return TMS_ERR_INVALID_ARG;
    if (n_tokens > 0 && (!doc_tokens || !aligned16(doc_tokens))) return TMS_ERR_INVALID_ARG;
    if (n_cand == 0) return TMS_OK;
    DeviceInfo dev;
    tms_status st = current_device(&dev);
    if (st != TMS_OK) return st;

    dense::Args a{};
    a.offsets = doc_offsets;
    a.lengths = doc_lengths;
    a.cand_ids = cand_ids;
    a.cand_offsets = cand_offsets;
    a.out = out_scores;
    a.err = dev.err;
    a.budget = debug_wait_budget();
    a.fault = debug_fault();
    a.n_docs = n_docs;
    a.n_tokens = n_tokens;
    a.n_cand = n_cand;
    a.n_flat = n_cand;
    a.group = 0;
    a.n_queries = n_queries;
    a.nq = nq;
    a.bpc = (nq + 31) / 32;

    if (dtype == TMS_F32) {
        // split TF32 on the tensor cores; the exact CUDA-core kernel below
        // covers the shapes that plan_tc's rule leaves out
        a.nchunks = (d + dense::chunk_elems(dense::kTF32) - 1) / dense::chunk_elems(dense::kTF32);
        st = tune ? dense::tune_tc<1, false, dense::kTF32>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens,
                                                           a, stream, n_timed)
                  : dense::launch_tc<1, false, dense::kTF32>(dev, queries, dtype, n_queries, nq, d, doc_tokens,
                                                             n_tokens, a, stream);
        if (st != TMS_ERR_UNSUPPORTED) return st;
        const int smem = 32 * d * 4;
        if (smem > dev.max_smem_optin) return TMS_ERR_UNSUPPORTED;
        if (cudaFuncSetAttribute(dense::dense_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
            cudaSuccess)
            return launch_status(cudaErrorInvalidValue);
        const int64_t want = (n_cand + dense::kF32Warps - 1) / dense::kF32Warps;
        const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(dev.sm_count, want));
        return launch_status(launch_dependent(dense::dense_f32_kernel, dim3(static_cast<unsigned>(grid)),
                                              dim3(dense::kF32Warps * 32), static_cast<size_t>(smem), stream,
                                              static_cast<const float*>(queries),
                                              static_cast<const float*>(doc_tokens), a, d));
    }
    a.nchunks = (d + dense::chunk_elems(dense::kF16) - 1) / dense::chunk_elems(dense::kF16);
    return tune ? dense::tune_tc<1, false, dense::kF16>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, a,
                                                        stream, n_timed)
                : dense::launch_tc<1, false, dense::kF16>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens,
                                                          a, stream);
}

}  // namespace
}  // namespace tms

extern "C" tms_status tms_score_dense(const void* queries, tms_dtype dtype, int n_queries, int nq, int d,
                                      const void* doc_tokens, int64_t n_tokens, const int64_t* doc_offsets,
                                      const int32_t* doc_lengths, int64_t n_docs, const int32_t* cand_ids,
                                      const int64_t* cand_offsets, int64_t n_cand, float* out_scores,
                                      cudaStream_t stream) {
    return tms::score_dense(queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, doc_offsets, doc_lengths, n_docs,
                            cand_ids, cand_offsets, n_cand, out_scores, stream, false, nullptr);
}

extern "C" tms_status tms_tune_dense(const void* queries, tms_dtype dtype, int n_queries, int nq, int d,
                                     const void* doc_tokens, int64_t n_tokens, const int64_t* doc_offsets,
                                     const int32_t* doc_lengths, int64_t n_docs, const int32_t* cand_ids,
                                     const int64_t* cand_offsets, int64_t n_cand, float* out_scores,
                                     cudaStream_t stream, int* n_configs) {
    return tms::score_dense(queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, doc_offsets, doc_lengths, n_docs,
                            cand_ids, cand_offsets, n_cand, out_scores, stream, true, n_configs);
}

namespace tms {
namespace {

tms_status score_dense_shared(const void* queries, tms_dtype dtype, int n_queries, int nq, int d,
                              const void* doc_tokens, int64_t n_tokens, const int64_t* doc_offsets,
                              const int32_t* doc_lengths, int64_t n_docs, const int32_t* cand_ids, int64_t n_cand,
                              float* out_scores, cudaStream_t stream, bool tune, int* n_configs) {
    if (n_configs) *n_configs = 0;
    if (dtype != TMS_F16 && dtype != TMS_BF16 && dtype != TMS_F32) return TMS_ERR_INVALID_ARG;
    if (n_queries < 1 || n_queries > 4096 || nq < 1 || nq > 128 || d < 8 || d > 1024 || d % 8 != 0)
        return TMS_ERR_INVALID_ARG;
    if (dtype == TMS_F32 || nq > 32) return TMS_ERR_UNSUPPORTED;
    if (n_tokens < 0 || n_tokens >= (int64_t(1) << 31) || n_docs < 0 || n_cand < 0) return TMS_ERR_INVALID_ARG;
    if (!queries || !aligned16(queries)) return TMS_ERR_INVALID_ARG;
    if (n_cand > 0 && (!cand_ids || !out_scores || !aligned16(cand_ids) || !aligned16(out_scores)))
        return TMS_ERR_INVALID_ARG;
    if (n_docs > 0 && (!doc_offsets || !doc_lengths || !aligned16(doc_offsets) || !aligned16(doc_lengths)))
        return TMS_ERR_INVALID_ARG;
    if (n_tokens > 0 && (!doc_tokens || !aligned16(doc_tokens))) return TMS_ERR_INVALID_ARG;
    if (n_cand == 0) return TMS_OK;
    DeviceInfo dev;
    tms_status st = current_device(&dev);
    if (st != TMS_OK) return st;
    dense::Args a{};
    a.offsets = doc_offsets;
    a.lengths = doc_lengths;
    a.cand_ids = cand_ids;
    a.cand_offsets = nullptr;
    a.out = out_scores;
    a.err = dev.err;
    a.budget = debug_wait_budget();
    a.fault = debug_fault();
    a.n_docs = n_docs;
    a.n_tokens = n_tokens;
    a.n_cand = n_cand;
    a.n_queries = n_queries;
    a.nq = nq;
    a.nchunks = (d + dense::chunk_elems(dense::kF16) - 1) / dense::chunk_elems(dense::kF16);
    return dense::shared_run<dense::kF16>(dev, queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, a, stream, tune,
                                          n_configs);
}

}  // namespace
}  // namespace tms

extern "C" tms_status tms_score_dense_shared(const void* queries, tms_dtype dtype, int n_queries, int nq, int d,
                                             const void* doc_tokens, int64_t n_tokens, const int64_t* doc_offsets,
                                             const int32_t* doc_lengths, int64_t n_docs, const int32_t* cand_ids,
                                             int64_t n_cand, float* out_scores, cudaStream_t stream) {
    return tms::score_dense_shared(queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, doc_offsets, doc_lengths,
                                   n_docs, cand_ids, n_cand, out_scores, stream, false, nullptr);
}

extern "C" tms_status tms_tune_dense_shared(const void* queries, tms_dtype dtype, int n_queries, int nq, int d,
                                            const void* doc_tokens, int64_t n_tokens, const int64_t* doc_offsets,
                                            const int32_t* doc_lengths, int64_t n_docs, const int32_t* cand_ids,
                                            int64_t n_cand, float* out_scores, cudaStream_t stream, int* n_configs) {
    return tms::score_dense_shared(queries, dtype, n_queries, nq, d, doc_tokens, n_tokens, doc_offsets, doc_lengths,
                                   n_docs, cand_ids, n_cand, out_scores, stream, true, n_configs);
}
