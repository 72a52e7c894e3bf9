// Residual check of a GEMM on the GPU in binary64 (Freivalds 1977).
//
// For C = alpha A B + beta C0 (A M x K, B K x N, C0 and C M x N, all row-major
// binary32) and vectors x (N) and y (M), the two identities
//   C x   = alpha A (B x)   + beta C0 x        (right form)
//   y^T C = alpha (y^T A) B + beta y^T C0      (left form)
// hold exactly for the exact product.  Every entry of C enters both sides, so a wrong
// tile, row block or single entry changes the residual vectors
//   r = C x - beta C0 x - alpha A (B x),  s = y^T C - beta y^T C0 - alpha (y^T A) B
// by exactly that entry's error times x_j (row i of r) and y_i (column j of s), while
// the check reads each matrix once instead of forming the O(MNK) product.  Every
// product and sum here is binary64 (the binary32 inputs are exact in binary64), so the
// check adds ~1e-16 relative noise to what it measures.
//
// Kernels (all deterministic: fixed partition, fixed summation order, no atomics):
//   rowdot  out[i] = sum_j X[i][j] v[j] (and the same for a second matrix), one warp per
//           row, lanes stride the row in float4 steps, a fixed butterfly at the end;
//   coldot  out[j] = sum_i w[i] X[i][j] (and a second matrix), column strips of 256 x
//           row chunks, binary64 partials per chunk, then the chunks summed in order;
//   norms   both residual vectors, their 2-norms and max-norms against the reference sides'.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "gao_internal.h"

namespace gao {
namespace {

// The check is bound by the binary64 pipe, not by HBM: this part completes 1.7 binary64
// operations per clock and SM (measured: DFMA and DADD 1.68, binary32-to-binary64 conversion
// 1.99, on the same pipe), so an element's conversion cost as much as its multiply-add.  Hence
//  - widen() forms the binary64 value with integer operations (exact, same bits), which leaves
//    the pipe to the eight multiply-adds per element quadruple (A, B, C, C0, two forms each):
//    M = N = K = 4096 takes 134 M of them, 0.27 ms at that rate against 0.04 ms of HBM reads;
//  - small blocks, so that the last SMs to finish hold little more than the average (512 blocks
//    of eight rows put 4 on some SMs and 3 on others, 16 % over the mean; 2048 of two rows, 4 %);
//  - the norms spread over a cluster of eight SMs and the chunk sums over 64-thread blocks
//    (one SM's pipe took 28 us for 4096 entries' norms, 18 us for a chunk sum).
// Together 748 -> 343 us at that size.
constexpr int kRowdotThreads = 64;   // 2 rows per block
constexpr int kColThreads = 64;      // 4 columns per thread: 256-column strips
constexpr int kColStrip = 4 * kColThreads;
constexpr int kChunkStrip = 512;     // columns a row chunk's size is reckoned by (fixes the sums' order)
constexpr int kMaxColChunks = 64;    // row chunks of a column reduction
constexpr int kColAhead = 4;        // rows of a column reduction's loads in flight
constexpr int kFinishThreads = 64;
constexpr int kNormThreads = 1024;   // threads of one form's norms, over a cluster of kNormCtas blocks
constexpr int kNormCtas = 8;

// f in binary64, formed with integer operations: sign, exponent + 896, the fraction shifted;
// zeros keep their sign.  Subnormal values, infinities and NaNs go through the conversion.
__device__ __forceinline__ bool widen_special(float f) {
    const uint32_t u = __float_as_uint(f) << 1;
    return u - 1u < 0x00FFFFFFu || u >= 0xFF000000u;
}
__device__ __forceinline__ double widen_plain(float f) {
    const uint32_t b = __float_as_uint(f);
    const uint32_t hi = (uint32_t)((int32_t)b >> 3) & 0x8FFFFFFFu;
    return __hiloint2double((int)(hi + ((b << 1) != 0u ? 0x38000000u : 0u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(float f) { return widen_special(f) ? (double)f : widen_plain(f); }
// Four values at once, one branch for the special ones.
__device__ __forceinline__ void widen4(const float (&f)[4], double (&d)[4]) {
    if (widen_special(f[0]) || widen_special(f[1]) || widen_special(f[2]) || widen_special(f[3])) {
#pragma unroll
        for (int q = 0; q < 4; ++q) d[q] = (double)f[q];
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) d[q] = widen_plain(f[q]);
    }
}

// out[i] = sum_j X[i][j] v[j], and out2[i] = sum_j X2[i][j] v[j] when X2 is set.
template <bool TWO>
__global__ void __launch_bounds__(kRowdotThreads) rowdot_kernel(const float* __restrict__ X,
                                                                const float* __restrict__ X2, int64_t rows,
                                                                int64_t cols, const double* __restrict__ v,
                                                                double* __restrict__ out, double* __restrict__ out2,
                                                                int vec) {
    const int lane = threadIdx.x & 31;
    constexpr int kRows = kRowdotThreads / 32;
    for (int64_t i = (int64_t)blockIdx.x * kRows + (threadIdx.x >> 5); i < rows; i += (int64_t)gridDim.x * kRows) {
        const float* xr = X + i * cols;
        const float* xr2 = TWO ? X2 + i * cols : nullptr;
        double a = 0.0, b = 0.0;
        int64_t j0 = 0;
        if (vec) {
            const int64_t n4 = cols / 4;
            for (int64_t q = lane; q < n4; q += 32) {
                const float4 u = __ldg(reinterpret_cast<const float4*>(xr) + q);
                const double2 v01 = __ldg(reinterpret_cast<const double2*>(v) + 2 * q);
                const double2 v23 = __ldg(reinterpret_cast<const double2*>(v) + 2 * q + 1);
                const float uf[4] = {u.x, u.y, u.z, u.w};
                double ud[4];
                if constexpr (TWO) {
                    const float4 w = __ldg(reinterpret_cast<const float4*>(xr2) + q);
                    const float wf[4] = {w.x, w.y, w.z, w.w};
                    double wd[4];
                    widen4(wf, wd);
                    b = fma(wd[0], v01.x, b);
                    b = fma(wd[1], v01.y, b);
                    b = fma(wd[2], v23.x, b);
                    b = fma(wd[3], v23.y, b);
                }
                widen4(uf, ud);
                a = fma(ud[0], v01.x, a);
                a = fma(ud[1], v01.y, a);
                a = fma(ud[2], v23.x, a);
                a = fma(ud[3], v23.y, a);
            }
            j0 = n4 * 4;
        }
        for (int64_t j = j0 + lane; j < cols; j += 32) {
            const double vj = v[j];
            a = fma(widen(xr[j]), vj, a);
            if constexpr (TWO) b = fma(widen(xr2[j]), vj, b);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, off);
            if constexpr (TWO) b += __shfl_xor_sync(0xffffffffu, b, off);
        }
        if (lane == 0) {
            out[i] = a;
            if constexpr (TWO) out2[i] = b;
        }
    }
}

// Partial column sums over the rows of chunk blockIdx.y:
// part[chunk][j] = sum_{i in chunk} w[i] X[i][j] (part2 likewise for X2).
template <bool TWO>
__global__ void __launch_bounds__(kColThreads) coldot_partial_kernel(const float* __restrict__ X,
                                                                     const float* __restrict__ X2, int64_t rows,
                                                                     int64_t cols, const double* __restrict__ w,
                                                                     int64_t rows_per_chunk,
                                                                     double* __restrict__ part,
                                                                     double* __restrict__ part2, int vec) {
    const int64_t j0 = (int64_t)blockIdx.x * kColStrip + 4 * threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.y * rows_per_chunk;
    const int64_t r1 = std::min(rows, r0 + rows_per_chunk);
    double a[4] = {0.0, 0.0, 0.0, 0.0}, b[4] = {0.0, 0.0, 0.0, 0.0};
    if (j0 < cols) {
        const bool full = vec && j0 + 3 < cols;
        // kColAhead rows' loads go out before the first is used: the branch in widen4 would
        // otherwise leave one row in flight (48 us for a 4096 x 4096 matrix against 34)
        for (int64_t i0 = r0; i0 < r1; i0 += kColAhead) {
            float u[kColAhead][4], t[TWO ? kColAhead : 1][4];
            double wi[kColAhead];
#pragma unroll
            for (int k = 0; k < kColAhead; ++k) {
                const int64_t i = i0 + k < r1 ? i0 + k : i0;  // rows past the chunk are not added
                wi[k] = w[i];
                const float* xr = X + i * cols + j0;
                if (full) {
                    const float4 q = __ldg(reinterpret_cast<const float4*>(xr));
                    u[k][0] = q.x, u[k][1] = q.y, u[k][2] = q.z, u[k][3] = q.w;
                    if constexpr (TWO) {
                        const float4 q2 = __ldg(reinterpret_cast<const float4*>(X2 + i * cols + j0));
                        t[k][0] = q2.x, t[k][1] = q2.y, t[k][2] = q2.z, t[k][3] = q2.w;
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        u[k][c] = j0 + c < cols ? xr[c] : 0.0f;
                        if constexpr (TWO) t[k][c] = j0 + c < cols ? X2[i * cols + j0 + c] : 0.0f;
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < kColAhead; ++k) {
                if (i0 + k >= r1) break;
                double d[4];
                widen4(u[k], d);
#pragma unroll
                for (int c = 0; c < 4; ++c) a[c] = fma(wi[k], d[c], a[c]);
                if constexpr (TWO) {
                    widen4(t[k], d);
#pragma unroll
                    for (int c = 0; c < 4; ++c) b[c] = fma(wi[k], d[c], b[c]);
                }
            }
        }
    }
    double* pr = part + (int64_t)blockIdx.y * cols;
    double* pr2 = TWO ? part2 + (int64_t)blockIdx.y * cols : nullptr;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (j0 + c < cols) {
            pr[j0 + c] = a[c];
            if constexpr (TWO) pr2[j0 + c] = b[c];
        }
    }
}

// out[j] = sum over chunks, in chunk order, of part[chunk][j]; blockIdx.y = 1: part2 into out2.
__global__ void __launch_bounds__(kFinishThreads) coldot_finish_kernel(const double* __restrict__ part,
                                                                       const double* __restrict__ part2,
                                                                       int64_t cols, int chunks,
                                                                       double* __restrict__ out,
                                                                       double* __restrict__ out2) {
    constexpr int kAhead = 16;  // loads in flight
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= cols) return;
    const double* src = (blockIdx.y ? part2 : part) + j;
    double a = 0.0;
    int c = 0;
    for (; c + kAhead <= chunks; c += kAhead) {
        double v[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) v[k] = src[(int64_t)(c + k) * cols];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) a += v[k];
    }
    for (; c < chunks; ++c) a += src[(int64_t)c * cols];
    (blockIdx.y ? out2 : out)[j] = a;
}

// One form's vectors: for n entries ref = alpha p + beta q0, res = c - beta q0 - alpha p (c =
// C's side); res written to rvec when set; norms[0] = ||res||_2, norms[1] = ||ref||_2,
// norms[2] = max |res|, norms[3] = max |ref|, norms[4] = the first index of max |res|.
struct NormForm {
    const double* c;
    const double* q0;
    const double* p;
    int64_t n;
    double* rvec;
    double* norms;
};

// Each form on a cluster of kNormCtas blocks (form = cluster index): kNormThreads threads
// stride the entries, a fixed butterfly within each warp, the warps' values gathered in the
// first block's shared memory and combined there in warp order, each quantity by its own warp.
__global__ void __cluster_dims__(kNormCtas, 1, 1) __launch_bounds__(kNormThreads / kNormCtas)
    residual_norms_kernel(NormForm right, NormForm left, double alpha, double beta) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int kWarps = kNormThreads / 32, kCtaThreads = kNormThreads / kNormCtas;
    __shared__ double s_rr[kWarps], s_ff[kWarps], s_rm[kWarps], s_fm[kWarps];
    __shared__ int64_t s_ri[kWarps];
    const NormForm& F = blockIdx.x < kNormCtas ? right : left;
    const int rank = (int)(blockIdx.x % kNormCtas), t = rank * kCtaThreads + (int)threadIdx.x;
    double rr = 0.0, ff = 0.0, rm = -1.0, fm = 0.0;
    int64_t ri = -1;
    for (int64_t i = t; i < F.n; i += kNormThreads) {
        const double ref = fma(alpha, F.p[i], beta * F.q0[i]);
        const double res = (F.c[i] - beta * F.q0[i]) - alpha * F.p[i];
        if (F.rvec) F.rvec[i] = res;
        rr = fma(res, res, rr);
        ff = fma(ref, ref, ff);
        if (fabs(res) > rm) rm = fabs(res), ri = i;  // first index of the maximum in this thread's order
        fm = fmax(fm, fabs(ref));
    }
    // fixed butterfly within the warp, then warps in order; the maximum keeps the lowest index
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        rr += __shfl_xor_sync(0xffffffffu, rr, off);
        ff += __shfl_xor_sync(0xffffffffu, ff, off);
        fm = fmax(fm, __shfl_xor_sync(0xffffffffu, fm, off));
        const double orm = __shfl_xor_sync(0xffffffffu, rm, off);
        const long long ori = __shfl_xor_sync(0xffffffffu, (long long)ri, off);
        if (orm > rm || (orm == rm && ori >= 0 && (ri < 0 || ori < ri))) rm = orm, ri = ori;
    }
    const int w = t >> 5;
    cluster.sync();  // every block of the cluster has started: its shared memory can be written
    if ((threadIdx.x & 31) == 0) {  // into the cluster's first block
        *cluster.map_shared_rank(s_rr + w, 0) = rr;
        *cluster.map_shared_rank(s_ff + w, 0) = ff;
        *cluster.map_shared_rank(s_rm + w, 0) = rm;
        *cluster.map_shared_rank(s_fm + w, 0) = fm;
        *cluster.map_shared_rank(s_ri + w, 0) = ri;
    }
    cluster.sync();
    if (rank != 0 || (threadIdx.x & 31) != 0) return;
    switch (threadIdx.x >> 5) {
        case 0: {
            double a = 0.0;
            for (int k = 0; k < kWarps; ++k) a += s_rr[k];
            F.norms[0] = sqrt(a);
            break;
        }
        case 1: {
            double f = 0.0;
            for (int k = 0; k < kWarps; ++k) f += s_ff[k];
            F.norms[1] = sqrt(f);
            break;
        }
        case 2: {
            double m = -1.0;
            int64_t mi = -1;
            for (int k = 0; k < kWarps; ++k)
                if (s_rm[k] > m || (s_rm[k] == m && s_ri[k] >= 0 && (mi < 0 || s_ri[k] < mi))) m = s_rm[k], mi = s_ri[k];
            F.norms[2] = m < 0.0 ? 0.0 : m;
            F.norms[4] = (double)mi;
            break;
        }
        case 3: {
            double mf = 0.0;
            for (int k = 0; k < kWarps; ++k) mf = fmax(mf, s_fm[k]);
            F.norms[3] = mf;
            break;
        }
    }
}

inline size_t a256(size_t x) { return (x + 255) / 256 * 256; }

int col_chunks(int64_t rows, int64_t cols) {
    // about four blocks per SM over the whole reduction, at most kMaxColChunks chunks
    const int64_t strips = (cols + kChunkStrip - 1) / kChunkStrip;
    int64_t c = (4 * (int64_t)sm_count() + strips - 1) / std::max<int64_t>(1, strips);
    c = std::max<int64_t>(1, std::min<int64_t>({c, (int64_t)kMaxColChunks, std::max<int64_t>(1, rows)}));
    return (int)c;
}

struct ResidLayout {
    size_t bx, abx, cx, c0x, ya, yab, yc, yc0, part, part2, norms, total;
};

ResidLayout resid_layout(int64_t M, int64_t N, int64_t K) {
    ResidLayout L{};
    const size_t d = sizeof(double);
    // partial sums of the three column reductions: y^T A (K columns), (y^T A) B and y^T C (N)
    const size_t part = std::max({(size_t)col_chunks(M, K) * (size_t)K, (size_t)col_chunks(K, N) * (size_t)N,
                                  (size_t)col_chunks(M, N) * (size_t)N});
    const size_t part2 = (size_t)col_chunks(M, N) * (size_t)N;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off += a256(std::max<size_t>(bytes, d));
        return o;
    };
    L.bx = take((size_t)K * d);
    L.abx = take((size_t)M * d);
    L.cx = take((size_t)M * d);
    L.c0x = take((size_t)M * d);
    L.ya = take((size_t)K * d);
    L.yab = take((size_t)N * d);
    L.yc = take((size_t)N * d);
    L.yc0 = take((size_t)N * d);
    L.part = take(part * d);
    L.part2 = take(part2 * d);
    L.norms = take(16 * d);
    L.total = off;
    return L;
}

cudaError_t launch_rowdot(const float* X, const float* X2, int64_t rows, int64_t cols, const double* v, double* out,
                          double* out2, cudaStream_t st) {
    if (rows <= 0) return cudaSuccess;
    const int vec = (cols % 4 == 0) && ((((uintptr_t)X) | ((uintptr_t)X2) | ((uintptr_t)v)) & 15u) == 0;
    const int64_t blocks = std::min<int64_t>((rows + kRowdotThreads / 32 - 1) / (kRowdotThreads / 32), 0x7fffffff);
    if (X2) rowdot_kernel<true><<<(unsigned)blocks, kRowdotThreads, 0, st>>>(X, X2, rows, cols, v, out, out2, vec);
    else rowdot_kernel<false><<<(unsigned)blocks, kRowdotThreads, 0, st>>>(X, nullptr, rows, cols, v, out, nullptr, vec);
    return cudaGetLastError();
}

cudaError_t launch_coldot(const float* X, const float* X2, int64_t rows, int64_t cols, const double* w, double* part,
                          double* part2, double* out, double* out2, cudaStream_t st) {
    if (cols <= 0) return cudaSuccess;
    const int chunks = col_chunks(rows, cols);
    const int64_t rpc = (std::max<int64_t>(rows, 1) + chunks - 1) / chunks;
    const int vec = (cols % 4 == 0) && ((((uintptr_t)X) | ((uintptr_t)X2)) & 15u) == 0;
    const dim3 grid((unsigned)((cols + kColStrip - 1) / kColStrip), (unsigned)chunks);
    if (X2) coldot_partial_kernel<true><<<grid, kColThreads, 0, st>>>(X, X2, rows, cols, w, rpc, part, part2, vec);
    else coldot_partial_kernel<false><<<grid, kColThreads, 0, st>>>(X, nullptr, rows, cols, w, rpc, part, nullptr, vec);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const dim3 fgrid((unsigned)((cols + kFinishThreads - 1) / kFinishThreads), X2 ? 2 : 1);
    coldot_finish_kernel<<<fgrid, kFinishThreads, 0, st>>>(part, part2, cols, chunks, out, out2);
    return cudaGetLastError();
}

}  // namespace

size_t gemm_residual_scratch_bytes(int64_t M, int64_t N, int64_t K) { return resid_layout(M, N, K).total; }

cudaError_t launch_gemm_residual(const float* A, const float* B, const float* C0, const float* C, int64_t M,
                                 int64_t N, int64_t K, double alpha, double beta, const double* x, const double* y,
                                 void* scratch, double* rvec, double* svec, cudaStream_t st, int* launches,
                                 const double** norms_dev) {
    const ResidLayout L = resid_layout(M, N, K);
    char* s = static_cast<char*>(scratch);
    auto D = [&](size_t off) { return reinterpret_cast<double*>(s + off); };
    double *bx = D(L.bx), *abx = D(L.abx), *cx = D(L.cx), *c0x = D(L.c0x), *ya = D(L.ya), *yab = D(L.yab),
           *yc = D(L.yc), *yc0 = D(L.yc0), *part = D(L.part), *part2 = D(L.part2), *norms = D(L.norms);
    *launches = 0;
    const bool has_c0 = C0 != nullptr && beta != 0.0;
    const float* c0 = has_c0 ? C0 : nullptr;
    cudaError_t e;
    // right form: B x, A (B x), C x and C0 x
    if (K > 0) {
        if ((e = launch_rowdot(B, nullptr, K, N, x, bx, nullptr, st)) != cudaSuccess) return e;
        if ((e = launch_rowdot(A, nullptr, M, K, bx, abx, nullptr, st)) != cudaSuccess) return e;
        *launches += 2;
    } else {
        if ((e = cudaMemsetAsync(abx, 0, (size_t)std::max<int64_t>(M, 1) * sizeof(double), st)) != cudaSuccess)
            return e;
    }
    if ((e = launch_rowdot(C, c0, M, N, x, cx, c0x, st)) != cudaSuccess) return e;
    if (!has_c0 && (e = cudaMemsetAsync(c0x, 0, (size_t)std::max<int64_t>(M, 1) * sizeof(double), st)) != cudaSuccess)
        return e;
    *launches += 1;
    // left form: y^T A, (y^T A) B, y^T C and y^T C0
    if (K > 0) {
        if ((e = launch_coldot(A, nullptr, M, K, y, part, nullptr, ya, nullptr, st)) != cudaSuccess) return e;
        if ((e = launch_coldot(B, nullptr, K, N, ya, part, nullptr, yab, nullptr, st)) != cudaSuccess) return e;
        *launches += 4;
    } else {
        if ((e = cudaMemsetAsync(yab, 0, (size_t)std::max<int64_t>(N, 1) * sizeof(double), st)) != cudaSuccess)
            return e;
    }
    if ((e = launch_coldot(C, c0, M, N, y, part, part2, yc, yc0, st)) != cudaSuccess) return e;
    if (!has_c0 && (e = cudaMemsetAsync(yc0, 0, (size_t)std::max<int64_t>(N, 1) * sizeof(double), st)) != cudaSuccess)
        return e;
    const NormForm right{cx, c0x, abx, M, rvec, norms}, left{yc, yc0, yab, N, svec, norms + 8};
    residual_norms_kernel<<<2 * kNormCtas, kNormThreads / kNormCtas, 0, st>>>(right, left, alpha, has_c0 ? beta : 0.0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *launches += 3;
    if (norms_dev) *norms_dev = norms;
    return cudaSuccess;
}

void residual_from_norms(const double* nr, gao_residual* out) {
    out->right = nr[1] > 0.0 ? nr[0] / nr[1] : nr[0];
    out->right_inf = nr[3] > 0.0 ? nr[2] / nr[3] : nr[2];
    out->right_argmax = (int64_t)nr[4];
    out->left = nr[9] > 0.0 ? nr[8] / nr[9] : nr[8];
    out->left_inf = nr[11] > 0.0 ? nr[10] / nr[11] : nr[10];
    out->left_argmax = (int64_t)nr[12];
}

}  // namespace gao

extern "C" gao_status gao_gemm_residual_scratch(int64_t M, int64_t N, int64_t K, uint64_t* bytes) {
    using namespace gao;
    if (!bytes) return fail(GAO_EINVAL, "bytes is null");
    if (M < 1 || N < 1 || K < 0) return fail(GAO_EINVAL, "gao_gemm_residual_scratch: M, N >= 1 and K >= 0");
    *bytes = gemm_residual_scratch_bytes(M, N, K);
    return GAO_OK;
}

extern "C" gao_status gao_gemm_residual(const float* A, const float* B, const float* C0, const float* C, int64_t M,
                                        int64_t N, int64_t K, double alpha, double beta, const double* x,
                                        const double* y, void* scratch, uint64_t scratch_bytes, double* r_out,
                                        double* s_out, gao_residual* out, void* stream) {
    using namespace gao;
    if (!out) return fail(GAO_EINVAL, "gao_gemm_residual: out is null");
    if (M < 1 || N < 1 || K < 0) return fail(GAO_EINVAL, "gao_gemm_residual: M, N >= 1 and K >= 0");
    if (!C || !x || !y || !scratch || (K > 0 && (!A || !B)))
        return fail(GAO_EINVAL, "gao_gemm_residual: null device pointer");
    if (scratch_bytes < gemm_residual_scratch_bytes(M, N, K) || ((uintptr_t)scratch & 255u))
        return fail(GAO_EINVAL, "gao_gemm_residual: scratch too small or not 256-byte aligned");
    if (M > (1LL << 40) || N > (1LL << 40) || K > (1LL << 40))
        return fail(GAO_EINVAL, "gao_gemm_residual: dimension too large");
    gao_status s = check_device(nullptr);
    if (s != GAO_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    double h[16];
    const double* nd = nullptr;
    int launches = 0;
    cudaError_t e = launch_gemm_residual(A, B, C0, C, M, N, K, alpha, beta, x, y, scratch, r_out, s_out, st,
                                         &launches, &nd);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, nd, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "gao_gemm_residual");
    residual_from_norms(h, out);
    return GAO_OK;
}
