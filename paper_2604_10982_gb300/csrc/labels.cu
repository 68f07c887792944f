// Per-surfel instance labels (Sec. 4.1, Eqs. 4-7) on the tensor cores.
//
// For surfel g (feature f_g, centre p_g) and instance query q (feature f_q,
// spatial Gaussian N(mu_q, Sigma_q)):
//     S(q, g) = sigmoid(f_q^T f_g)                                   (Eq. 4)
//     D(q, g) = phi_q(p_g) / phi_q(mu_q)
//             = exp(-(p_g - mu_q)^T Sigma_q^-1 (p_g - mu_q) / 2)      (Eq. 5)
//     l(g)    = softmax over q of S D                            (Eqs. 6-7)
// The dot products f_q^T f_g run in the row-tile tcgen05 pipeline
// (rowgemm.cuh: 128 surfels per tile, the queries resident in shared
// memory, FP32 accumulation in TMEM). The epilogue keeps each surfel's row of
// dot products in registers and applies the sigmoid, the geometric factor
// and the softmax in FP32; the queries' centres and precision matrices
// (inverted from Sigma once per CTA) sit in shared memory. With 8 epilogue
// warps per SM the kernel is bound by the latency of a row's arithmetic, so 16
// queries are worked on at a time without a branch between them (columns past
// n_q are computed on zeroed query data and masked) and the row leaves in
// 16-byte stores: 811 -> 494 us for 1M surfels, 100 queries, D = 128. The label table
// [n, ld] is written in FP32 or BF16 with zero columns past n_q, so it can be
// rendered like a feature table (Eq. 8).
#include <cuda_bf16.h>

#include "rowgemm.cuh"

namespace psi {
namespace {

using namespace tc;

constexpr int kQP = 12; // floats per query in shared memory: mu (3), precision (6), pad
// Row g of a [n, ld] table in BF16 or FP32 (ld a multiple of 16): columns
// below n_q from A * scale, zero past it. 16-byte stores (a warp's 4-byte
// stores would each touch 32 sectors).
__device__ __forceinline__ void store_row(void *table, int64_t g, int ld, int n_q, bool bf16, const float *A, float scale)
{
    auto at = [&](int q) { return q < n_q ? A[q] * scale : 0.0f; };
    if (bf16) {
        uint4 *row = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(table) + g * ld);
#pragma unroll
        for (int q = 0; q < static_cast<int>(kRowAccStride); q += 8)
            if (q < ld) {
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const __nv_bfloat162 p2 = __floats2bfloat162_rn(at(q + 2 * k), at(q + 2 * k + 1));
                    w[k] = *reinterpret_cast<const uint32_t *>(&p2);
                }
                row[q >> 3] = make_uint4(w[0], w[1], w[2], w[3]);
            }
    } else {
        float4 *row = reinterpret_cast<float4 *>(static_cast<float *>(table) + g * ld);
#pragma unroll
        for (int q = 0; q < static_cast<int>(kRowAccStride); q += 4)
            if (q < ld) row[q >> 2] = make_float4(at(q), at(q + 1), at(q + 2), at(q + 3));
    }
}

struct LabelEpi {
    static constexpr int kStages = 2; // two CTAs per SM: the softmax epilogue dominates
    int64_t n;
    int n_q;
    const float *centres; // [n, 3]
    const float *q_mu;    // [n_q, 3]
    const float *q_cov;   // [n_q, 6]: xx, xy, xz, yy, yz, zz
    void *labels;         // [n, ld]
    int ld;
    int out_bf16;

    struct Pre {
        float x, y, z;
    };

    // each query's centre and precision Sigma^-1 (adjugate over determinant);
    // zero past n_q
    __device__ __forceinline__ void prepare(unsigned char *smem, int tid) const
    {
        float *s = reinterpret_cast<float *>(smem);
        for (int q = tid; q < static_cast<int>(kRowAccStride); q += kRowThreads) {
            float *o = s + kQP * q;
            if (q >= n_q) {
                for (int k = 0; k < kQP; ++k) o[k] = 0.0f;
                continue;
            }
            const float a = q_cov[6 * q], b = q_cov[6 * q + 1], c = q_cov[6 * q + 2];
            const float d = q_cov[6 * q + 3], e = q_cov[6 * q + 4], f = q_cov[6 * q + 5];
            const float A11 = d * f - e * e, A12 = c * e - b * f, A13 = b * e - c * d;
            const float A22 = a * f - c * c, A23 = b * c - a * e, A33 = a * d - b * b;
            const float inv = 1.0f / (a * A11 + b * A12 + c * A13);
            o[0] = q_mu[3 * q];
            o[1] = q_mu[3 * q + 1];
            o[2] = q_mu[3 * q + 2];
            o[3] = A11 * inv;
            o[4] = A12 * inv;
            o[5] = A13 * inv;
            o[6] = A22 * inv;
            o[7] = A23 * inv;
            o[8] = A33 * inv;
        }
    }

    __device__ __forceinline__ Pre begin(int64_t g) const
    {
        if (g >= n) return Pre{0.f, 0.f, 0.f};
        return Pre{__ldg(centres + 3 * g), __ldg(centres + 3 * g + 1), __ldg(centres + 3 * g + 2)};
    }

    // scores are computed in place over the row of dot products (r)
    __device__ __forceinline__ void end(int64_t g, uint32_t (&r)[kRowAccStride], Pre p, bool fail,
                                        unsigned char *smem) const
    {
        if (g >= n || fail) return;
        const float4 *s = reinterpret_cast<const float4 *>(smem);
        float *A = reinterpret_cast<float *>(r);
        const float ninf = -__int_as_float(0x7f800000);
        float amax = ninf;
#pragma unroll
        for (int q0 = 0; q0 < static_cast<int>(kRowAccStride); q0 += 16) {
            if (q0 >= n_q) break;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int q = q0 + k;
                const float4 u = s[3 * q], v = s[3 * q + 1], w = s[3 * q + 2];
                const float o[9] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w, w.x};
                const float dx = p.x - o[0], dy = p.y - o[1], dz = p.z - o[2];
                const float m2 = o[3] * dx * dx + o[6] * dy * dy + o[8] * dz * dz +
                                 2.0f * (o[4] * dx * dy + o[5] * dx * dz + o[7] * dy * dz);
                const float S = 1.0f / (1.0f + __expf(-A[q]));
                A[q] = q < n_q ? S * __expf(-0.5f * m2) : ninf;
                amax = fmaxf(amax, A[q]);
            }
        }
        float sum = 0.0f;
#pragma unroll
        for (int q0 = 0; q0 < static_cast<int>(kRowAccStride); q0 += 16) {
            if (q0 >= n_q) break;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                A[q0 + k] = __expf(A[q0 + k] - amax); // 0 past n_q
                sum += A[q0 + k];
            }
        }
        const float inv = 1.0f / sum;
        store_row(labels, g, ld, n_q, out_bf16, A, inv);
    }
};

// The plain per-surfel query logits f_q^T f_g (no sigmoid, geometric factor
// or softmax): composited with the Top-K weights they give, by linearity,
// the decode's logits <F, q> of every pixel without forming F.
struct LogitEpi {
    static constexpr int kStages = 4; // one CTA per SM: bound by the table's stores
    int64_t n;
    int n_q;
    void *table; // [n, ld]
    int ld;
    int out_bf16;

    struct Pre {};
    __device__ __forceinline__ void prepare(unsigned char *, int) const {}
    __device__ __forceinline__ Pre begin(int64_t) const { return Pre{}; }
    __device__ __forceinline__ void end(int64_t g, uint32_t (&r)[kRowAccStride], Pre, bool fail, unsigned char *) const
    {
        if (g >= n || fail) return;
        store_row(table, g, ld, n_q, out_bf16, reinterpret_cast<const float *>(r), 1.0f);
    }
};

} // namespace

cudaError_t launch_logits(const void *F, int64_t n, int D, const void *Q, int n_q, void *table, int ld, int out_bf16,
                          DevStatus *status, cudaStream_t st, const char **why)
{
    const LogitEpi epi{n, n_q, table, ld, out_bf16};
    return launch_row_gemm(F, n, D, Q, n_q, 0, epi, status, st, why);
}

cudaError_t launch_labels(const void *F, int64_t n, int D, const float *centres, const void *Q, int n_q,
                          const float *q_mu, const float *q_cov, void *labels, int ld, int out_bf16, DevStatus *status,
                          cudaStream_t st, const char **why)
{
    const LabelEpi epi{n, n_q, centres, q_mu, q_cov, labels, ld, out_bf16};
    return launch_row_gemm(F, n, D, Q, n_q, static_cast<size_t>(kQP) * 128 * sizeof(float), epi, status, st, why);
}

} // namespace psi
