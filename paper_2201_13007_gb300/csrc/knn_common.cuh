// knn_common.cuh -- what the brute-force k-NN kernels share: the key
// encoding, the legacy tensor-core product whose FP32 sums define a key, row
// norms, cp.async staging.
#pragma once

#include <cuda_bf16.h>

#include "knn.cuh"

namespace ann {
namespace {

constexpr int KBM = 128;  // query rows per CTA
constexpr unsigned long long KMAX = ~0ull;

__device__ __forceinline__ uint32_t ord_enc(float f) {
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ __forceinline__ float ord_dec(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Four 8x8 BF16 matrices; lane i names row i % 8 of matrix i / 8.
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t saddr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(saddr));
}

__device__ __forceinline__ void cp_async16(uint32_t saddr, const void *gmem, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(saddr), "l"(gmem), "r"(valid ? 16 : 0)
                 : "memory");
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Pitch of a staged BF16 row: 8 elements more than the row, so that the eight
// rows of an ldmatrix land in different banks.
__host__ __device__ constexpr int knn_pitch(int d) { return d + 8; }

// Squared norm of a BF16 row in FP32, elements added in order.
__device__ __forceinline__ float bf16_norm(const __nv_bfloat16 *x, int d) {
    float acc = 0.f;
    for (int i = 0; i < d; i += 8) {  // d is a multiple of 32 and rows start on 16 bytes
        const uint4 w = *reinterpret_cast<const uint4 *>(x + i);
        const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float lo = __uint_as_float(u[j] << 16), hi = __uint_as_float(u[j] & 0xFFFF0000u);
            acc = fmaf(lo, lo, acc);
            acc = fmaf(hi, hi, acc);
        }
    }
    return acc;
}

// The key of one (query, base row) pair from their product v, the base
// row's norm bn and the query's norm qn.
template <bool L2>
__device__ __forceinline__ float knn_dist(float v, float bn, float qn) {
    return L2 ? fmaxf(fmaf(-2.f, v, bn) + qn, 0.f) : -v;
}

}  // namespace
}  // namespace ann
