// FP32 matrix product on the CUDA cores, C = scale A B with gathered rows (fold.h).
//
// Bound by the FP32 pipes: a thread keeps TM x TN sums and reads TM + TN shared values per
// k, in 16-byte loads whose lanes fall in distinct banks or on the same address. The sums
// go two columns at a time through fma.rn.f32x2, which leaves half the issue slots to the
// loads and to the duplication of the A values (the FMA rate is the same as that of scalar
// FMAs, and so are the roundings).
#include <algorithm>

#include "f32x2.cuh"
#include "fold.h"
#include "tc_ptx.cuh"

namespace mpiffl {

namespace {

constexpr int kSgK = 16;  // K per stage, two stages

// 16 bytes global -> shared, the last 16 - n of them zero
__device__ __forceinline__ void cp_async16(void *dst, const void *src, int n) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(n)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

struct SgemmBatch {
    SgemmArgs g[kSgemmMax];
    int first[kSgemmMax + 1];  // first block of each problem
};

// K of one run of sums: longer products add their runs' sums, so that rounding errors grow
// with the run and the number of runs, not with K
constexpr int kSgRun = 256;

// One BM x BN tile per block. A warp covers 8 row groups x 4 column groups: its A loads
// take 8 distinct 16-byte units side by side (a thread's rows come in runs of 4, BM / (TM / 4)
// rows apart), its B loads 4.
template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN)) k_sgemm(const __grid_constant__ SgemmBatch batch) {
    constexpr int T = (BM / TM) * (BN / TN);
    constexpr int LA = BM + 4;
    constexpr int NA = (BM * kSgK / 4 + T - 1) / T, NB = (BN * kSgK / 4 + T - 1) / T;
    static_assert(BM / TM == 8 && TM % 4 == 0 && TN % 4 == 0 && T % 32 == 0, "warp layout");
    __shared__ __align__(16) float sA[2][kSgK][LA];
    __shared__ __align__(16) float sB[2][kSgK][BN];
    int pi = 0;
    while ((int)blockIdx.x >= batch.first[pi + 1]) ++pi;  // uniform
    const SgemmArgs &g = batch.g[pi];
    const int b = (int)blockIdx.x - batch.first[pi];
    const int ntn = (g.N + BN - 1) / BN;
    const int m0 = b / ntn * BM, c0 = b % ntn * BN;
    const int tid = threadIdx.x, lane = tid & 31;
    const int tr = lane >> 2, tc = (tid >> 5) * 4 + (lane & 3);

    // the rows this thread loads: row (tid + u T) mod BM, K quad (tid + u T) / BM
    const float *ap[NA];
#pragma unroll
    for (int u = 0; u < NA; ++u) {
        const int i = tid + u * T, r = m0 + i % BM;
        const bool in = i < BM * kSgK / 4 && r < g.M;
        ap[u] = in ? g.A + (size_t)(g.arow ? __ldg(g.arow + r) : r) * g.lda : nullptr;
    }
    const bool vec = !g.acol && g.lda % 4 == 0 && (reinterpret_cast<uintptr_t>(g.A) & 15) == 0;
    float4 ra[NA];
    auto load_a = [&](int k0) {
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            const int k = k0 + 4 * ((tid + u * T) / BM);
            ra[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (ap[u]) {
                if (vec && k + 4 <= g.K) {
                    ra[u] = __ldg(reinterpret_cast<const float4 *>(ap[u] + k));
                } else {
                    auto at = [&](int kk) {
                        return kk < g.K ? __ldg(ap[u] + (g.acol ? __ldg(g.acol + kk) : kk)) : 0.f;
                    };
                    ra[u] = make_float4(at(k), at(k + 1), at(k + 2), at(k + 3));
                }
            }
        }
    };
    auto store_a = [&](int s) {
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            const int i = tid + u * T, r = i % BM, kq = 4 * (i / BM);
            if (i < BM * kSgK / 4) {
                sA[s][kq][r] = ra[u].x;
                sA[s][kq + 1][r] = ra[u].y;
                sA[s][kq + 2][r] = ra[u].z;
                sA[s][kq + 3][r] = ra[u].w;
            }
        }
    };
    auto copy_b = [&](int k0, int s) {
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int i = tid + u * T, kk = i / (BN / 4), c = 4 * (i % (BN / 4));
            if (i < BN * kSgK / 4) {
                const bool in = k0 + kk < g.K && c0 + c < g.ldb;
                cp_async16(&sB[s][kk][c], in ? g.B + (size_t)(k0 + kk) * g.ldb + c0 + c : g.B, in ? 16 : 0);
            }
        }
    };

    f32x2 acc[TM][TN / 2], sum[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = sum[i][j] = 0;
    copy_b(0, 0);
    ptx::grid_dep_wait();  // A comes from the previous kernel
    ptx::grid_dep_launch();
    load_a(0);
    store_a(0);
    cp_async_wait();
    __syncthreads();
    const int nk = (g.K + kSgK - 1) / kSgK;
    for (int t = 0; t < nk; ++t) {
        const int s = t & 1;
        if (t + 1 < nk) {
            copy_b((t + 1) * kSgK, s ^ 1);
            load_a((t + 1) * kSgK);
        }
#pragma unroll
        for (int kk = 0; kk < kSgK; ++kk) {
            f32x2 bv[TN / 2];
#pragma unroll
            for (int j = 0; j < TN / 4; ++j) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&sB[s][kk][j * (BN / (TN / 4)) + 4 * tc]);
                bv[2 * j] = v.x;
                bv[2 * j + 1] = v.y;
            }
#pragma unroll
            for (int i = 0; i < TM / 4; ++i) {
                const float4 a4 = *reinterpret_cast<const float4 *>(&sA[s][kk][i * (BM / (TM / 4)) + 4 * tr]);
                const float av[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const f32x2 a2 = dup2(av[q]);
#pragma unroll
                    for (int j = 0; j < TN / 2; ++j) acc[4 * i + q][j] = fma2(a2, bv[j], acc[4 * i + q][j]);
                }
            }
        }
        if (t + 1 < nk) {
            store_a(s ^ 1);
            cp_async_wait();
        }
        if ((t + 1) % (kSgRun / kSgK) == 0 || t + 1 == nk) {
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) {
                    sum[i][j] = add2(sum[i][j], acc[i][j]);
                    acc[i][j] = 0;
                }
        }
        __syncthreads();
    }
    const bool vecc = !g.ccol && g.ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(g.C) & 15) == 0;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int r = m0 + (i / 4) * (BM / (TM / 4)) + 4 * tr + (i & 3);
        if (r >= g.M) continue;
        const float sc = g.scale ? __ldg(g.scale + (g.arow ? __ldg(g.arow + r) : r) / g.rdiv) : 1.f;
        float *dst = g.C + (size_t)(g.crow ? __ldg(g.crow + r) : r) * g.ldc;
#pragma unroll
        for (int j = 0; j < TN / 4; ++j) {
            const int c = c0 + j * (BN / (TN / 4)) + 4 * tc;
            const float2 lo = unpack2(sum[i][2 * j]), hi = unpack2(sum[i][2 * j + 1]);
            const float4 v = make_float4(sc * lo.x, sc * lo.y, sc * hi.x, sc * hi.y);
            if (vecc && c + 4 <= g.N) {
                *reinterpret_cast<float4 *>(dst + c) = v;
            } else {
                const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (c + q < g.N) dst[g.ccol ? __ldg(g.ccol + c + q) : c + q] = e[q];
            }
        }
    }
}

template <int BM, int BN, int TM, int TN>
void run(const SgemmArgs *g, int n, cudaStream_t st) {
    SgemmBatch b{};
    for (int i = 0; i < kSgemmMax; ++i) {
        const int tiles = i < n ? (g[i].M + BM - 1) / BM * ((g[i].N + BN - 1) / BN) : 0;
        if (i < n) b.g[i] = g[i];
        b.first[i + 1] = b.first[i] + tiles;
    }
    const int total = b.first[kSgemmMax];
    if (total > 0)
        launch_dependent(k_sgemm<BM, BN, TM, TN>, dim3(total), dim3((BM / TM) * (BN / TN)), 0, st, b);
}

}  // namespace

void launch_sgemm(const SgemmArgs *g, int n, cudaStream_t st) {
    // 64 x 96 tiles where they fill the GPU; smaller ones, with more blocks, where not
    long long big = 0;
    for (int i = 0; i < n; ++i) big += (long long)((g[i].M + 63) / 64) * ((g[i].N + 95) / 96);
    if (big >= 100) run<64, 96, 8, 4>(g, n, st);
    else run<32, 32, 4, 4>(g, n, st);
}

}  // namespace mpiffl
