// FP32 matrix product on the CUDA cores, C = scale A B with gathered rows (fold.h).
//
// Bound by the FP32 pipes: a thread keeps TM x TN sums and reads TM + TN shared values per
// k, in 16-byte loads whose lanes fall in distinct banks or on the same address. The sums
// go two columns at a time through fma.rn.f32x2, which leaves half the issue slots to the
// loads and to the duplication of the A values (the FMA rate is the same as that of scalar
// FMAs, and so are the roundings).
#include <algorithm>

#include "fold.h"
#include "tc_ptx.cuh"

namespace mpiffl {

namespace {

constexpr int kSgK = 16;  // K per stage, two stages

using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 dup2(float a) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

// 16 bytes global -> shared, the last 16 - n of them zero
__device__ __forceinline__ void cp_async16(void *dst, const void *src, int n) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(n)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One BM x BN tile per block. A warp covers 8 row groups x 4 column groups: its A loads
// take 8 distinct 16-byte units side by side (a thread's rows come in runs of 4, BM / (TM / 4)
// rows apart), its B loads 4.
template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN)) k_sgemm(SgemmArgs g0, SgemmArgs g1, int n0) {
    constexpr int T = (BM / TM) * (BN / TN);
    constexpr int LA = BM + 4;
    constexpr int NA = (BM * kSgK / 4 + T - 1) / T, NB = (BN * kSgK / 4 + T - 1) / T;
    static_assert(BM / TM == 8 && TM % 4 == 0 && TN % 4 == 0 && T % 32 == 0, "warp layout");
    __shared__ __align__(16) float sA[2][kSgK][LA];
    __shared__ __align__(16) float sB[2][kSgK][BN];
    const bool second = (int)blockIdx.x >= n0;
    const SgemmArgs g = second ? g1 : g0;
    const int b = (int)blockIdx.x - (second ? n0 : 0);
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
    const bool vec = g.lda % 4 == 0 && (reinterpret_cast<uintptr_t>(g.A) & 15) == 0;
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
                    if (k < g.K) ra[u].x = __ldg(ap[u] + k);
                    if (k + 1 < g.K) ra[u].y = __ldg(ap[u] + k + 1);
                    if (k + 2 < g.K) ra[u].z = __ldg(ap[u] + k + 2);
                    if (k + 3 < g.K) ra[u].w = __ldg(ap[u] + k + 3);
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

    f32x2 acc[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0;
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
        __syncthreads();
    }
    const bool vecc = g.ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(g.C) & 15) == 0;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int r = m0 + (i / 4) * (BM / (TM / 4)) + 4 * tr + (i & 3);
        if (r >= g.M) continue;
        const float sc = g.scale ? __ldg(g.scale + (g.arow ? __ldg(g.arow + r) : r) / g.rdiv) : 1.f;
        float *dst = g.C + (size_t)(g.crow ? __ldg(g.crow + r) : r) * g.ldc;
#pragma unroll
        for (int j = 0; j < TN / 4; ++j) {
            const int c = c0 + j * (BN / (TN / 4)) + 4 * tc;
            const float2 lo = unpack2(acc[i][2 * j]), hi = unpack2(acc[i][2 * j + 1]);
            const float4 v = make_float4(sc * lo.x, sc * lo.y, sc * hi.x, sc * hi.y);
            if (vecc && c + 4 <= g.N) {
                *reinterpret_cast<float4 *>(dst + c) = v;
            } else {
                if (c < g.N) dst[c] = v.x;
                if (c + 1 < g.N) dst[c + 1] = v.y;
                if (c + 2 < g.N) dst[c + 2] = v.z;
                if (c + 3 < g.N) dst[c + 3] = v.w;
            }
        }
    }
}

template <int BM, int BN, int TM, int TN>
void run(const SgemmArgs *g, int n, cudaStream_t st) {
    auto tiles = [](const SgemmArgs &a) { return (a.M + BM - 1) / BM * ((a.N + BN - 1) / BN); };
    const int n0 = tiles(g[0]), n1 = n > 1 ? tiles(g[1]) : 0;
    if (n0 + n1 == 0) return;
    launch_dependent(k_sgemm<BM, BN, TM, TN>, dim3(n0 + n1), dim3((BM / TM) * (BN / TN)), 0, st, g[0],
                     g[n > 1 ? 1 : 0], n0);
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
