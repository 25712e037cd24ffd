// knn.cuh -- the brute-force k-NN over BF16 rows, for the host side.
#pragma once

#include "ann_internal.cuh"

namespace ann {

// knn_filter.cu: brute-force k-NN over BF16 rows (graph construction). A plan
// gives the workspace a call needs (one device allocation, offsets of its
// parts) and how the base and the queries are cut.
struct KnnPlan {
    int levels;        // the base is taken in levels + 1 nested samples
    int chunk_blocks;  // blocks of 128 query rows per pass over the base
    int splits;        // CTAs that share a block's tiles
    int no_loads;      // 0; 1 = the filter's waits run out (tests)
    size_t err, norms, bias, over, qnorm, margin, thr, kept_n, counts, kept, lists, bytes;
};
KnnPlan knn_plan(int64_t n, int64_t nq, int sms);
// The int at ws + plan.err is set if a wait (2) or a merge (1) ran out; the kernels after that do nothing.
cudaError_t launch_knn_bf16(const KnnPlan &plan, void *ws, const void *base, int64_t n, int d, const void *queries,
                            int64_t nq, int64_t self0, int metric, int k, int32_t *ids, float *dists, int sms,
                            cudaStream_t stream);
// The same by the scan kernel alone, for small calls (knn_scan_is_faster) and
// callers without room for the plan's workspace: ws holds knn_scan_bytes(n);
// its first int is the error word.
bool knn_scan_is_faster(int64_t n, int64_t nq);
size_t knn_scan_bytes(int64_t n);
cudaError_t launch_knn_scan_all(void *ws, const void *base, int64_t n, int d, const void *queries, int64_t nq,
                                int64_t self0, int metric, int k, int32_t *ids, float *dists, cudaStream_t stream);
// knn.cu: the scan kernel, for the blocks of 128 query rows with only[block]
// set (all if only is null). norms holds the base rows' squared norms (zeros up to
// knn_norms_rows(n)); err is set to 1 if a CTA's merge rounds ran out, and nothing is done by a CTA that finds it set.
int64_t knn_norms_rows(int64_t n);
cudaError_t launch_knn_scan(const void *base, int64_t n, int d, const void *queries, int64_t nq, int64_t self0,
                            int metric, int k, int32_t *ids, float *dists, const float *norms, const int *only,
                            int *err, cudaStream_t stream);

}  // namespace ann
