// FP32 SIMT GEMM on the CUDA cores: C = alpha * A @ B + beta * C0.
//
// The "plain FP32" path; A and B are row-major (A: M x K, B: K x N).
//
// Accuracy: a single binary32 accumulator over a long K grows its rounding error with K, so
// the K loop is split into chunks of `kchunk` elements; each chunk is summed from zero in
// registers and the chunk sums are then added in order.  Every element takes the same
// operations in the same order whatever the tile and the split, and as the host loop does, so
// all give the same bits.
//
// What bounds it: the FP32 lanes (128 multiply-adds per clock and SM) and, next to them, shared
// memory, which returns 128 bytes per clock and SM: with an 8 x 8 register tile per thread the
// operand reads take as many clocks as the multiply-adds (that kernel reached 0.61 of the
// lanes), with 8 x 16 three quarters of them.  Packed multiply-adds (fma.rn.f32x2: two columns
// of a row, the same rounding per element) leave the issue slots that the loads, the operand
// duplication and the loop need.  Both operands go to shared memory by cp.async (no register
// staging): A as rows of BK elements (a thread reads four k of a row at once), B as it lies; on the
// large tiles, where rows are not 16-byte aligned, through registers (RAG).
// A small problem has too few tiles to fill the GPU; since the chunks are summed apart anyway, a
// cluster can split them (no order changes), and smaller tiles serve where that is not enough.
// Measured, n x n x n, us between events (before: 128 x 128 tiles of 8 x 8 per thread, scalar FFMAs):
//   n = 256: 45 -> 13, 1000: 148 -> 62, 1001: 156 -> 69, 2048: 432 -> 350, 2049: 485 -> 465, 4096: 3028 ->
//   2490 (55 of 80 TFLOP/s).  What is left: two warps per scheduler issue a packed multiply-add every
//   other clock with little to cover the operand reads, and the last wave of tiles.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "gao_internal.h"

namespace gao {
namespace {

// TM x TN elements per thread; a warp is 4 x 8 threads; WM x WN warps form the block tile.
template <int TM_, int TN_, int WM_, int WN_, int BK_, int STAGES_, int MINB_>
struct Shape {
    static constexpr int TM = TM_, TN = TN_, WM = WM_, WN = WN_, BK = BK_, STAGES = STAGES_, MINB = MINB_;
    static constexpr int THREADS = 32 * WM * WN;
    static constexpr int BM = WM * 4 * TM, BN = WN * 8 * TN;
    static constexpr int LDA = BK + 4;  // rows of A 16 bytes apart in banks: four rows read at once without conflicts
    static constexpr int A_FLOATS = BM * LDA, B_FLOATS = BK * BN;  // one stage
    static constexpr int E = TM * TN / 4;                          // groups of four columns per thread
    static constexpr size_t TILE_BYTES = (size_t)STAGES * (A_FLOATS + B_FLOATS) * 4;
    static constexpr size_t SUM_BYTES = (size_t)E * THREADS * 16;  // running sums, or a split chunk's sums
};
using Large = Shape<8, 16, 4, 1, 16, 2, 2>;   // 128 x 128, 128 threads
using Medium = Shape<8, 8, 2, 1, 16, 3, 4>;   // 64 x 64, 64 threads
using Small = Shape<4, 4, 2, 1, 32, 4, 4>;    // 32 x 32, 64 threads

using f32x2 = unsigned long long;  // two binary32 values, the lower address in the low half

// acc = a * b + acc in both halves, one rounding each.
__device__ __forceinline__ void ffma2(f32x2& acc, f32x2 a, f32x2 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 unpack(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 dup(float a) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
}
// BYTES from global to shared memory without passing through registers; zeros where !in.
template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const float* src, bool in) {
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0) : "memory");
}

// va, vb, vc: rows of A; of B; of C and C0 are 16-byte aligned.  SPLIT: a cluster of
// ceil(K / kc) blocks along z shares a tile, each summing one chunk; the sums meet in shared
// memory and each block adds, in chunk order, and stores its share of the tile.
// RAG: both operands go through registers, a word at a time and a step ahead, where cp.async would
// move a word an instruction and lane: that cost the large tiles more than their loads' latency
// (INIT and GEMM, us, cp.async -> registers: 2049^3 532 -> 483, 3001^3 1474 -> 1405, 8001 x 801 x 601
// 257 -> 241; 256 threads of 8 x 8 before: 498, 1419, 259; only K of a few steps is better off with
// cp.async, 5000 x 5000 x 33 120 -> 128, before 163).
template <class S, bool SPLIT, bool RAG>
__global__ void __launch_bounds__(S::THREADS, S::MINB)
    sgemm_kernel(float* C, const float* __restrict__ A, const float* __restrict__ B, const float* C0, int64_t M,
                 int64_t N, int64_t K, float alpha, float beta, int64_t kc, bool va, bool vb, bool vc) {
    constexpr int TM = S::TM, TN = S::TN, BK = S::BK, THREADS = S::THREADS;
    extern __shared__ __align__(16) float smem[];
    float* As = smem;                                        // [STAGES][BM][LDA]
    float* Bs = smem + S::STAGES * S::A_FLOATS;              // [STAGES][BK][BN]
    float4* ssum = reinterpret_cast<float4*>(smem + S::STAGES * (S::A_FLOATS + S::B_FLOATS));  // [E][THREADS]
    const uint32_t as_addr = (uint32_t)__cvta_generic_to_shared(As);
    const uint32_t bs_addr = (uint32_t)__cvta_generic_to_shared(Bs);
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int wm = w / S::WN, wn = w % S::WN, ty = lane >> 3, tx = lane & 7;
    const int64_t m0 = (int64_t)blockIdx.y * S::BM, n0 = (int64_t)blockIdx.x * S::BN;
    // this block's part of K: everything, or one chunk
    const int64_t kbeg = SPLIT ? (int64_t)blockIdx.z * kc : 0;
    const int64_t kend = SPLIT && kbeg + kc < K ? kbeg + kc : K;
    const int64_t nk = (kend - kbeg + BK - 1) / BK;
    const bool one = SPLIT || K <= kc;  // a single chunk: its sums are not added to anything here

    auto load = [&](int64_t kt) {
        const int st = (int)(kt % S::STAGES);
        const int64_t k0 = kbeg + kt * BK;
        const uint32_t a_dst = as_addr + (uint32_t)(st * S::A_FLOATS) * 4, b_dst = bs_addr + (uint32_t)(st * S::B_FLOATS) * 4;
        if (va) {
#pragma unroll
            for (int i = 0; i < S::BM * BK / 4 / THREADS; ++i) {
                const int e = i * THREADS + t, r = e / (BK / 4), c = e % (BK / 4) * 4;
                const bool in = m0 + r < M && k0 + c < kend;
                cp_async<16>(a_dst + (uint32_t)(r * S::LDA + c) * 4, in ? A + (m0 + r) * K + k0 + c : A, in);
            }
        } else {
#pragma unroll 4
            for (int i = 0; i < S::BM * BK / THREADS; ++i) {
                const int e = i * THREADS + t, r = e / BK, c = e % BK;
                const bool in = m0 + r < M && k0 + c < kend;
                cp_async<4>(a_dst + (uint32_t)(r * S::LDA + c) * 4, in ? A + (m0 + r) * K + k0 + c : A, in);
            }
        }
        if (vb) {
#pragma unroll
            for (int i = 0; i < BK * S::BN / 4 / THREADS; ++i) {
                const int e = i * THREADS + t, r = e / (S::BN / 4), c = e % (S::BN / 4) * 4;
                const bool in = k0 + r < kend && n0 + c < N;
                cp_async<16>(b_dst + (uint32_t)(r * S::BN + c) * 4, in ? B + (k0 + r) * N + n0 + c : B, in);
            }
        } else {
#pragma unroll 4
            for (int i = 0; i < BK * S::BN / THREADS; ++i) {
                const int e = i * THREADS + t, r = e / S::BN, c = e % S::BN;
                const bool in = k0 + r < kend && n0 + c < N;
                cp_async<4>(b_dst + (uint32_t)(r * S::BN + c) * 4, in ? B + (k0 + r) * N + n0 + c : B, in);
            }
        }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    constexpr int RA = RAG ? S::BM * BK / THREADS : 1, RB = RAG ? BK * S::BN / THREADS : 1;
    float ra[RA], rb[RB];
    auto fetch = [&](int64_t kt) {
        const int64_t k0 = kbeg + kt * BK;
#pragma unroll
        for (int i = 0; i < RA; ++i) {
            const int e = i * THREADS + t, r = e / BK, c = e % BK;
            ra[i] = m0 + r < M && k0 + c < kend ? __ldg(A + (m0 + r) * K + k0 + c) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int e = i * THREADS + t, r = e / S::BN, c = e % S::BN;
            rb[i] = k0 + r < kend && n0 + c < N ? __ldg(B + (k0 + r) * N + n0 + c) : 0.0f;
        }
    };
    auto put = [&](int64_t kt) {
        float* as = As + (int)(kt % S::STAGES) * S::A_FLOATS;
        float* bs = Bs + (int)(kt % S::STAGES) * S::B_FLOATS;
#pragma unroll
        for (int i = 0; i < RA; ++i) as[(i * THREADS + t) / BK * S::LDA + (i * THREADS + t) % BK] = ra[i];
#pragma unroll
        for (int i = 0; i < RB; ++i) bs[i * THREADS + t] = rb[i];
    };

    f32x2 acc[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
    // group e = (row i, column quad h) of this thread's sums
    auto group = [&](int i, int h) {
        const float2 u = unpack(acc[i][2 * h]), v = unpack(acc[i][2 * h + 1]);
        return make_float4(u.x, u.y, v.x, v.y);
    };
    if (!one) {
#pragma unroll
        for (int e = 0; e < S::E; ++e) ssum[e * THREADS + t] = make_float4(0, 0, 0, 0);
    }

    if constexpr (RAG) {
        if (nk > 0) {
            fetch(0);
            put(0);
        }
    } else {
#pragma unroll
        for (int s = 0; s < S::STAGES - 1; ++s) {
            if (s < nk) load(s);
            commit();
        }
    }
    const int64_t chunk_tiles16 = kc / 16;  // 16-element steps per chunk
    int64_t left = chunk_tiles16;
    for (int64_t kt = 0; kt < nk; ++kt) {
        if constexpr (!RAG) asm volatile("cp.async.wait_group %0;" ::"n"(S::STAGES - 2) : "memory");
        __syncthreads();  // stage kt has landed for every thread; everyone is done with stage kt - 1
        if constexpr (RAG) {
            if (kt + 1 < nk) fetch(kt + 1);
        } else {
            if (kt + S::STAGES - 1 < nk) load(kt + S::STAGES - 1);
            commit();
        }
        const int st = (int)(kt % S::STAGES);
        const float* as = As + st * S::A_FLOATS + (wm * 4 * TM + ty) * S::LDA;  // rows ty, ty + 4, ...
        const float* bs = Bs + st * S::B_FLOATS + wn * 8 * TN + tx * 4;         // column quads 32 apart
#pragma unroll 1
        for (int g = 0; g < BK / 16; ++g) {  // 16 elements of K
            // fragments one step ahead of their use: B's of the next k, A's of the next pair of k
            float2 fa[2][TM];
            f32x2 fb[2][TN / 2];
            auto load_a = [&](int k2, float2 (&d)[TM]) {
#pragma unroll
                for (int i = 0; i < TM; ++i)
                    d[i] = *reinterpret_cast<const float2*>(as + i * 4 * S::LDA + g * 16 + 2 * k2);
            };
            auto load_b = [&](int k, f32x2 (&d)[TN / 2]) {
#pragma unroll
                for (int h = 0; h < TN / 4; ++h) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(bs + (g * 16 + k) * S::BN + h * 32);
                    d[2 * h] = v.x;
                    d[2 * h + 1] = v.y;
                }
            };
            load_a(0, fa[0]);
            load_b(0, fb[0]);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                if (k + 1 < 16) load_b(k + 1, fb[(k + 1) & 1]);
                if (k % 2 == 0 && k + 2 < 16) load_a(k / 2 + 1, fa[(k / 2 + 1) & 1]);
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    const float2 v = fa[(k / 2) & 1][i];
                    const f32x2 aa = dup(k % 2 ? v.y : v.x);
#pragma unroll
                    for (int j = 0; j < TN / 2; ++j) ffma2(acc[i][j], aa, fb[k & 1][j]);
                }
            }
            if (!one) {
                // a chunk (a multiple of 16 elements) is complete, or K is (steps past K hold
                // zeros and change nothing)
                left -= 1;
                if (left == 0 || (kt + 1 == nk && g + 1 == BK / 16)) {
                    left = chunk_tiles16;
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int h = 0; h < TN / 4; ++h) {
                            const float4 v = group(i, h);
                            float4& s = ssum[(i * (TN / 4) + h) * THREADS + t];
                            float4 x = s;
                            x.x += v.x, x.y += v.y, x.z += v.z, x.w += v.w;
                            s = x;
                            acc[i][2 * h] = acc[i][2 * h + 1] = 0ull;
                        }
                }
            }
        }
        if constexpr (RAG) {
            if (kt + 1 < nk) put(kt + 1);  // its stage was last read before this step's barrier
        }
    }

    // group e of thread t: its place in C, its C0, and alpha times its sums plus beta C0, stored.  C may
    // be C0, so a load waits for the stores before it: a row's groups are read before the first
    // of them is stored (one at a time made 5000 x 5000 x 33 take 184 us; 162 with 256 threads)
    auto row_of = [&](int e) { return m0 + wm * 4 * TM + e / (TN / 4) * 4 + ty; };
    auto col_of = [&](int e) { return n0 + wn * 8 * TN + e % (TN / 4) * 32 + tx * 4; };
    auto read_c0 = [&](int e) {
        const int64_t gm = row_of(e), gn = col_of(e);
        float4 c = make_float4(0, 0, 0, 0);
        if (beta == 0.0f || gm >= M || gn >= N) return c;
        const float* p = C0 + gm * N + gn;
        if (vc) return *reinterpret_cast<const float4*>(p);
        c.x = p[0];
        if (gn + 1 < N) c.y = p[1];
        if (gn + 2 < N) c.z = p[2];
        if (gn + 3 < N) c.w = p[3];
        return c;
    };
    auto finish = [&](int e, float4 s, float4 c) {
        const int64_t gm = row_of(e), gn = col_of(e);
        if (gm >= M || gn >= N) return;
        float r[4] = {alpha * s.x, alpha * s.y, alpha * s.z, alpha * s.w};
        if (beta != 0.0f) {
            r[0] = fmaf(beta, c.x, r[0]);
            r[1] = fmaf(beta, c.y, r[1]);
            r[2] = fmaf(beta, c.z, r[2]);
            r[3] = fmaf(beta, c.w, r[3]);
        }
        if (vc) {
            *reinterpret_cast<float4*>(C + gm * N + gn) = make_float4(r[0], r[1], r[2], r[3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (gn + q < N) C[gm * N + gn + q] = r[q];
        }
    };
    if constexpr (SPLIT) {
        namespace cg = cooperative_groups;
        cg::cluster_group cluster = cg::this_cluster();
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int h = 0; h < TN / 4; ++h) ssum[(i * (TN / 4) + h) * THREADS + t] = group(i, h);
        cluster.sync();
        const int nb = (int)gridDim.z, rank = (int)blockIdx.z;
        for (int e = rank; e < S::E; e += nb) {
            const float4 c = read_c0(e);
            float4 x = make_float4(0, 0, 0, 0);
            for (int j = 0; j < nb; ++j) {
                const float4 v = *cluster.map_shared_rank(&ssum[e * THREADS + t], j);
                x.x += v.x, x.y += v.y, x.z += v.z, x.w += v.w;
            }
            finish(e, x, c);
        }
        cluster.sync();  // no block leaves while another still reads its sums
    } else {
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            float4 c[TN / 4];
#pragma unroll
            for (int h = 0; h < TN / 4; ++h) c[h] = read_c0(i * (TN / 4) + h);
#pragma unroll
            for (int h = 0; h < TN / 4; ++h) {
                const int e = i * (TN / 4) + h;
                if (one) {  // + 0: the sums start at +0
                    const float4 v = group(i, h);
                    finish(e, make_float4(0.0f + v.x, 0.0f + v.y, 0.0f + v.z, 0.0f + v.w), c[h]);
                } else {
                    finish(e, ssum[e * THREADS + t], c[h]);
                }
            }
        }
    }
}

template <class S, bool SPLIT, bool RAG>
cudaError_t launch_shape(float* C, const float* A, const float* B, const float* C0, int64_t M, int64_t N, int64_t K,
                         float alpha, float beta, int64_t kc, cudaStream_t st) {
    auto kern = sgemm_kernel<S, SPLIT, RAG>;
    constexpr int most = (int)(S::TILE_BYTES + S::SUM_BYTES);
    static bool attr_set = false;  // per instantiation
    if (!attr_set) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    auto al = [](const void* p) { return ((uintptr_t)p & 15u) == 0; };
    const bool va = K % 4 == 0 && al(A), vb = N % 4 == 0 && al(B), vc = N % 4 == 0 && al(C) && al(C0);
    const unsigned nb = SPLIT ? (unsigned)((K + kc - 1) / kc) : 1u;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)((N + S::BN - 1) / S::BN), (unsigned)((M + S::BM - 1) / S::BM), nb);
    lc.blockDim = dim3(S::THREADS);
    lc.dynamicSmemBytes = S::TILE_BYTES + (SPLIT || K > kc ? S::SUM_BYTES : 0);
    lc.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 1;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = nb;
    lc.attrs = &at;
    lc.numAttrs = SPLIT ? 1 : 0;
    return cudaLaunchKernelEx(&lc, kern, C, A, B, C0, M, N, K, alpha, beta, kc, va, vb, vc);
}

}  // namespace

cudaError_t launch_gemm_simt(float* C, const float* A, const float* B, const float* C0, int64_t M, int64_t N,
                             int64_t K, float alpha, float beta, int kchunk, cudaStream_t st, double beside) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    if ((M + 127) / 128 > 65535) return cudaErrorInvalidValue;
    const int64_t kc = kchunk > 0 ? (((int64_t)kchunk + 15) / 16) * 16 : (int64_t)1 << 40;  // above any K: one chunk
    // The shape, and whether a cluster splits the chunks (2 to 8 of them), with the least
    // estimated time: the fullest SM holds u blocks, which take max(lat, u w) clocks per element
    // of K (lat: a block alone, bound by latency; w: its share of a busy SM), plus a fixed cost
    // (launch, first loads, a split's exchange).  The figures are fits to times measured over
    // n = 128 .. 4096 (within 10 %); rows that are not 16-byte aligned cost `ragged` more.  A GEMM
    // that shares the GPU with others' is taken to have its part of the SMs, since the small tiles'
    // extra loads then cost all of them (whole batches, us, as if alone / so / 128 x 128 tiles of 256
    // threads for all: 20 programs of 100 to 2000 rows, unaligned, 1930 / 1847 / 1790, aligned 1532 /
    // 1519 / 1622; eight of 512 to 1024, unaligned, 494 / 428 / 475).
    struct Model {
        int tile;
        double lat, w, fixed, fixed_split, ragged;
    };
    static constexpr Model kModel[3] = {{128, 218, 185, 6e3, 20e3, 1.36},
                                        {64, 140, 55, 6e3, 11e3, 1.53},
                                        {32, 58, 19, 6e3, 9e3, 1.7}};
    const bool rows16 = K % 4 == 0 && N % 4 == 0 && ((((uintptr_t)A) | ((uintptr_t)B)) & 15u) == 0;
    const int64_t chunks = (K + kc - 1) / kc;
    const int64_t sms = std::max<int64_t>(1, (int64_t)(sm_count() / std::max(1.0, beside)));
    int best = 0;
    double least = 0.0;
    for (int i = 0; i < 6; ++i) {
        const Model& m = kModel[i >> 1];
        const bool split = i & 1;
        const int64_t tm = (M + m.tile - 1) / m.tile, tn = (N + m.tile - 1) / m.tile;
        if (tm > 65535 || (split && (chunks < 2 || chunks > 8))) continue;
        const int64_t blocks = tm * tn * (split ? chunks : 1);
        const double u = (double)((blocks + sms - 1) / sms);
        const double per_k = std::max(m.lat, u * m.w) * (rows16 ? 1.0 : m.ragged);
        const double cost = per_k * (double)(split ? kc : K) + (split ? m.fixed_split : m.fixed);
        if (i == 0 || cost < least) {
            least = cost;
            best = i;
        }
    }
#define GAO_SIMT(S, SPLIT, RAG) launch_shape<S, SPLIT, RAG>(C, A, B, C0, M, N, K, alpha, beta, kc, st)
    switch (best) {
        case 0: return rows16 ? GAO_SIMT(Large, false, false) : GAO_SIMT(Large, false, true);
        case 1: return rows16 ? GAO_SIMT(Large, true, false) : GAO_SIMT(Large, true, true);
        case 2: return GAO_SIMT(Medium, false, false);
        case 3: return GAO_SIMT(Medium, true, false);
        case 4: return GAO_SIMT(Small, false, false);
        default: return GAO_SIMT(Small, true, false);
    }
#undef GAO_SIMT
}

}  // namespace gao
