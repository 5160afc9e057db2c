// FP32 matrix product on the CUDA cores, C = scale A B with gathered rows (fold.h).
//
// Bound by the FP32 pipes and by shared-memory loads together: a thread keeps TM x TN sums
// and reads TM + TN shared values per k, A four k at a time. The sums go two columns at a
// time through fma.rn.f32x2, which leaves half the issue slots to the loads and to the
// duplication of the A values. Both operands come through a ring of four stages filled
// by cp.async, so that a stage's latency (about a microsecond) is spread over three.
#include <algorithm>

#include "f32x2.cuh"
#include "fold.h"
#include "tc_ptx.cuh"

namespace mpiffl {

namespace {

constexpr int kSgK = 16;
// stages of the ring: three where sums wait in shared memory, so that three blocks fit an SM
__host__ __device__ constexpr int sg_stages(int mode) { return mode ? 3 : 4; }
constexpr int kSgRow = kSgK + 4;  // floats of a staged A row: 8 rows start in distinct bank groups

// 16 bytes global -> shared, the last 16 - n of them zero
__device__ __forceinline__ void cp_async16(void *dst, const void *src, int n) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(n)
                 : "memory");
}
// 4 bytes, zero when n is 0
__device__ __forceinline__ void cp_async4(void *dst, const void *src, int n) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(n)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

struct SgemmBatch {
    SgemmArgs g[kSgemmMax];
    int run;                   // K of one run of sums
    int first[kSgemmMax + 1];  // first block of each problem
};

// K of one run of sums (a multiple of kSgK): longer products add their runs' sums, so that rounding
// errors grow with the run and the number of runs, not with K. The shorter run is that of fine
// products in large tiles.
constexpr int kSgRun = 320, kSgRunFine = 64;

// One BM x BN tile per block. A warp covers 8 row groups x 4 column groups of TM x TN sums
// each (a thread's rows are 8 apart, its columns come in runs of 4, BN / (TN / 4) apart). A
// 16-byte shared load takes two cycles where neighbouring lanes share the address (the A
// loads here), four where they do not (B). KG: groups of threads that take their share of
// each stage's K and add their sums at the end (more warps for products with few tiles).
// MODE 1: K above kSgRun, the runs' sums are added in shared memory. MODE 2: two products of
// half values of k each; the first one's sums wait there for the second's. FINE: the sums of a
// stage are formed apart and then added, which takes a second set of registers.
__host__ __device__ constexpr int sgemm_stage_floats(int BM, int BN) { return BM * kSgRow + kSgK * BN; }
__host__ __device__ constexpr int sgemm_ring_floats(int BM, int BN, int join, int stages) {
    const int ring = stages * sgemm_stage_floats(BM, BN);
    return ring > join ? ring : join;
}

template <int BM, int BN, int TM, int TN, int KG, int MODE, bool FINE = false>
__global__ void __launch_bounds__((BM / TM) * (BN / TN) * KG, 384 / ((BM / TM) * (BN / TN) * KG))
    k_sgemm(const __grid_constant__ SgemmBatch batch) {
    constexpr int TG = (BM / TM) * (BN / TN), T = TG * KG;
    constexpr int NA = (BM * kSgK / 4 + T - 1) / T, NB = (BN * kSgK / 4 + T - 1) / T;
    constexpr int KS = kSgK / KG;
    constexpr int kStage = sgemm_stage_floats(BM, BN), kSgStages = sg_stages(MODE);
    static_assert(BM / TM == 8 && TN % 4 == 0 && TG % 32 == 0 && KS % 4 == 0, "warp layout");
    // the ring (the groups' sums take its place at the end), then MODE > 0: float2 [TM][TN / 2][T]
    extern __shared__ __align__(16) float smf[];
    float2 *sum = reinterpret_cast<float2 *>(smf + sgemm_ring_floats(BM, BN, (KG - 1) * TG * TM * TN, kSgStages));
    int pi = 0;
    while ((int)blockIdx.x >= batch.first[pi + 1]) ++pi;  // uniform
    const SgemmArgs &g = batch.g[pi];
    const int ntn = (g.N + BN - 1) / BN, nt = (g.M + BM - 1) / BM * ntn;
    const int bi = ((int)blockIdx.x - batch.first[pi]) / nt, b = (int)blockIdx.x - batch.first[pi] - bi * nt;
    const int m0 = b / ntn * BM, c0 = b % ntn * BN;
    const float *gA = g.A + bi * g.sA, *gB = g.B + bi * g.sB;
    const int bcols = g.bcols ? g.bcols : g.ldb;
    const int tid = threadIdx.x, lane = tid & 31, kg = tid / TG;
    const int tr = lane >> 2, tc = (tid % TG >> 5) * 4 + (lane & 3);

    // This thread's part of a stage of A: K quad tid mod 4 of the rows tid / 4 + u T / 4. Past
    // the last row the tile's rows again, whose sums are not stored (not one row for all of
    // them: copies of one address to many places take turns, 64 rows in tiles of 56 took three
    // times as long).
    static_assert(T % (kSgK / 4) == 0 && T % (BN / 4) == 0, "a thread keeps its K quad and its columns");
    const int ka = 4 * (tid % (kSgK / 4));
    const float *ap[NA];
#pragma unroll
    for (int u = 0; u < NA; ++u) {
        const int r = m0 + (tid + u * T) / (kSgK / 4) % min(BM, g.M - m0);
        ap[u] = gA + (size_t)(g.arow ? __ldg(g.arow + r) : r) * g.lda;
    }
    const bool vec = !g.acol && g.lda % 4 == 0 && (reinterpret_cast<uintptr_t>(gA) & 15) == 0;
    const int Kv = MODE == 2 ? g.half : g.K, th = (Kv + kSgK - 1) / kSgK;  // values and stages of a product
    // first value of stage t: k0 + t kstep (a product in halves counts its own)
    const int kstep = MODE != 2 && g.back ? -kSgK : kSgK, k0 = MODE != 2 && g.back ? (th - 1) * kSgK : 0;
    auto stage_k = [&](int t) { return MODE == 2 ? (t >= th ? t - th : t) * kSgK : k0 + t * kstep; };
    auto copy_a = [&](int t) {
        float *st = smf + (t % kSgStages) * kStage + (tid / (kSgK / 4)) * kSgRow + ka;
        const bool second = MODE == 2 && t >= th;
        const int k = stage_k(t) + ka, n = min(4, max(0, Kv - k));
        const int ks = min(k, (Kv - 1) & ~3) + (second ? g.ahalf : 0);
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            if ((BM * kSgK / 4) % T && tid + u * T >= BM * kSgK / 4) break;
            float *dst = st + u * (T / (kSgK / 4)) * kSgRow;
            if (vec) {
                cp_async16(dst, ap[u] + ks, 4 * n);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const bool in = k + e < Kv;
                    cp_async4(dst + e, in ? ap[u] + (MODE == 2 ? ks + e : g.acol ? __ldg(g.acol + k + e) : k + e) : gA,
                              in ? 4 : 0);
                }
            }
        }
    };
    // of B: columns cb of the rows tid / (BN / 4) + u T / (BN / 4)
    const int cb = c0 + 4 * (tid % (BN / 4)), kb0 = tid / (BN / 4);
    const float *bp = gB + min(cb, bcols - 4);
    const int kvalid = cb < bcols ? Kv : 0;
    auto copy_b = [&](int t) {
        float *st = smf + (t % kSgStages) * kStage + BM * kSgRow + 4 * tid;
        const bool second = MODE == 2 && t >= th;
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            if ((BN * kSgK / 4) % T && tid + u * T >= BN * kSgK / 4) break;
            const int kk = stage_k(t) + kb0 + u * (T / (BN / 4));
            cp_async16(st + 4 * u * T, bp + (int64_t)(min(kk, Kv - 1) + (second ? g.bhalf : 0)) * g.ldb,
                       kk < kvalid ? 16 : 0);
        }
    };

    // rows by pairs (2j, 2j + 1) of the thread's columns
    f32x2 acc[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0;
    const int nk = MODE == 2 ? 2 * th : th;
    ptx::grid_dep_wait();  // A comes from the previous kernel
    ptx::grid_dep_launch();
#pragma unroll
    for (int t = 0; t < kSgStages - 1; ++t) {
        if (t < nk) {
            copy_a(t);
            copy_b(t);
        }
        cp_async_commit();
    }
    for (int t = 0; t < nk; ++t) {
        cp_async_wait<kSgStages - 2>();
        __syncthreads();  // stage t has landed and stage t - 1 has been read
        if (t + kSgStages - 1 < nk) {
            copy_a(t + kSgStages - 1);
            copy_b(t + kSgStages - 1);
        }
        cp_async_commit();
        const float *st = smf + (t % kSgStages) * kStage;
        f32x2 part[FINE ? TM : 1][FINE ? TN / 2 : 1];  // sums of this stage
        const float *sa = st + tr * kSgRow + kg * KS, *sb = st + BM * kSgRow + kg * KS * BN + 4 * tc;
#pragma unroll
        for (int kb = 0; kb < KS; kb += 4) {
            float4 a4[TM];
#pragma unroll
            for (int i = 0; i < TM; ++i) a4[i] = *reinterpret_cast<const float4 *>(sa + 8 * i * kSgRow + kb);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                f32x2 bv[TN / 2];
#pragma unroll
                for (int j = 0; j < TN / 4; ++j) {
                    const ulonglong2 v =
                        *reinterpret_cast<const ulonglong2 *>(sb + (kb + q) * BN + j * (BN / (TN / 4)));
                    bv[2 * j] = v.x;
                    bv[2 * j + 1] = v.y;
                }
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    const f32x2 a2 = dup2(q == 0 ? a4[i].x : q == 1 ? a4[i].y : q == 2 ? a4[i].z : a4[i].w);
#pragma unroll
                    for (int j = 0; j < TN / 2; ++j)
                        if constexpr (FINE) part[i][j] = kb + q == 0 ? mul2(a2, bv[j]) : fma2(a2, bv[j], part[i][j]);
                        else acc[i][j] = fma2(a2, bv[j], acc[i][j]);
                }
            }
        }
        if constexpr (FINE)
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) acc[i][j] = add2(acc[i][j], part[i][j]);
        if (MODE == 2 && t + 1 == th)  // a thread's own words
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) {
                    sum[(i * (TN / 2) + j) * T + tid] = unpack2(acc[i][j]);
                    acc[i][j] = 0;
                }
        if (MODE == 1 && ((t + 1) % (batch.run * KG / kSgK) == 0 || t + 1 == nk)) {  // a thread's own words
            const bool first = t < batch.run * KG / kSgK;
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) {
                    float2 &w = sum[(i * (TN / 2) + j) * T + tid];
                    const float2 a = unpack2(acc[i][j]), o = first ? make_float2(0.f, 0.f) : w;
                    const float2 n = make_float2(o.x + a.x, o.y + a.y);
                    w = n;
                    acc[i][j] = t + 1 == nk ? pack2(n.x, n.y) : 0;
                }
        }
    }
    if (MODE == 2)  // E - O in its place in shared memory, E + O in registers
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN / 2; ++j) {
                float2 &w = sum[(i * (TN / 2) + j) * T + tid];
                const float2 o = unpack2(acc[i][j]), e = w;
                w = make_float2(e.x - o.x, e.y - o.y);
                acc[i][j] = pack2(e.x + o.x, e.y + o.y);
            }
    if (KG > 1) {  // group 0 adds the other groups' sums in their order
        __syncthreads();
        float2 *join = reinterpret_cast<float2 *>(smf);
        if (kg > 0)
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN / 2; ++j)
                    join[(((kg - 1) * TM + i) * (TN / 2) + j) * TG + tid % TG] = unpack2(acc[i][j]);
        __syncthreads();
        if (kg > 0) return;
        for (int q = 0; q < KG - 1; ++q)
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) {
                    const float2 o = join[((q * TM + i) * (TN / 2) + j) * TG + tid];
                    acc[i][j] = add2(acc[i][j], pack2(o.x, o.y));
                }
    }
    float *gC = g.C + bi * g.sC;
    const bool vecc = !g.ccol && g.ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(gC) & 15) == 0;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int r = m0 + tr + 8 * i;
        if (r >= g.M) continue;
        const float sc = g.scale ? __ldg(g.scale + (g.arow ? __ldg(g.arow + r) : r) / g.rdiv) : 1.f;
        float *dst = gC + (size_t)(g.crow ? __ldg(g.crow + r) : r) * g.ldc;
#pragma unroll
        for (int j = 0; j < TN / 4; ++j) {
            const int c = c0 + j * (BN / (TN / 4)) + 4 * tc;
            const float2 lo = unpack2(acc[i][2 * j]), hi = unpack2(acc[i][2 * j + 1]);
            const float e[4] = {sc * lo.x, sc * lo.y, sc * hi.x, sc * hi.y};
            if (vecc && c + 4 <= g.N) {
                *reinterpret_cast<float4 *>(dst + c) = make_float4(e[0], e[1], e[2], e[3]);
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (c + q < g.N) dst[g.ccol ? __ldg(g.ccol + c + q) : c + q] = e[q];
            }
            if (MODE == 2) {
                float d[4];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    float2 w = sum[(i * (TN / 2) + 2 * j + q) * T + tid];
                    for (int k = 1; k < KG; ++k) {
                        const float2 v = sum[(i * (TN / 2) + 2 * j + q) * T + k * TG + tid];
                        w = make_float2(w.x + v.x, w.y + v.y);
                    }
                    d[2 * q] = sc * w.x;
                    d[2 * q + 1] = sc * w.y;
                }
                const int c1 = g.mirror ? g.c1 - c - 3 : g.c1 + c;
                if (vecc && c + 4 <= g.N && c1 % 4 == 0) {
                    *reinterpret_cast<float4 *>(dst + c1) =
                        g.mirror ? make_float4(d[3], d[2], d[1], d[0]) : make_float4(d[0], d[1], d[2], d[3]);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (c + q < g.N) dst[g.mirror ? g.c1 - c - q : c1 + q] = d[q];
                }
            }
        }
    }
}

int batches(const SgemmArgs *g, int i, int n) { return i < n ? std::max(0, g[i].nbatch) : 0; }

template <int BM, int BN, int TM, int TN, int KG>
void run(const SgemmArgs *g, int n, cudaStream_t st) {
    constexpr int T = (BM / TM) * (BN / TN) * KG;
    SgemmBatch b{};
    const bool fine = g[0].fine;  // all products of one launch or none; the same for half
    b.run = fine && KG == 1 ? kSgRunFine : kSgRun;
    bool runs = false;
    for (int i = 0; i < kSgemmMax; ++i) {
        const int tiles = i < n ? (g[i].M + BM - 1) / BM * ((g[i].N + BN - 1) / BN) : 0;
        if (i < n) b.g[i] = g[i];
        if (i < n && (g[i].half > 0 || g[i].K > b.run * KG)) runs = true;
        b.first[i + 1] = b.first[i] + tiles * batches(g, i, n);
    }
    const int total = b.first[kSgemmMax];
    if (total == 0) return;
    const size_t smem = sizeof(float) * (sgemm_ring_floats(BM, BN, (KG - 1) * T / KG * TM * TN, sg_stages(runs)) + (runs ? TM * TN * T : 0));
    void (*kernel)(SgemmBatch);
    if constexpr (TM == 6) {  // fine halves alone
        kernel = k_sgemm<BM, BN, TM, TN, KG, 2, true>;
    } else {
        kernel = runs ? k_sgemm<BM, BN, TM, TN, KG, 1> : k_sgemm<BM, BN, TM, TN, KG, 0>;
        if constexpr (TM == 4)
            if (fine) kernel = runs ? k_sgemm<BM, BN, TM, TN, KG, 1, true> : k_sgemm<BM, BN, TM, TN, KG, 0, true>;
        if constexpr (TM == 4 || KG == 1)
            if (g[0].half > 0) kernel = k_sgemm<BM, BN, TM, TN, KG, 2>;
    }
    if (smem > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_dependent(kernel, dim3(total), dim3(T), smem, st, b);
}

}  // namespace

constexpr int kFineRows = 48;  // of a tile of fine halves

int sgemm_tiles(const SgemmArgs &g) {
    const int rows = g.fine && g.half > 0 ? kFineRows : 64;
    return (g.M + rows - 1) / rows * ((g.N + 127) / 128);
}

// 8 x 8 sums a thread (the fewest shared loads an FMA) where such tiles come to almost a wave
// of three blocks an SM: 4608 x 2304 x 256 in 106 us, 68% of the FP32 FMA rate (4 x 8 sums in
// 32 x 64 tiles and two groups along K: 129 us). Smaller products take the smaller tiles:
// 4608 x 288 x 256 in 22 us (29 us with the large tiles), 1536 x 168 x 128 in 5.5 us (11 us).
// Of the large tiles those of 56 rows where their waves are shorter: two halves of 4608 x 1152
// x 128 in 59 us (two waves of 64 rows, the second a third full: 67 us).
//
// Fine products (the z-drive adjoint's last one, over n_par W S values without an order of size):
// the small tiles have the registers for a stage's own sums, halves take them in tiles of 48 rows
// (those of 64 or 56 spill: the z-drive adjoint at 256^2 x 128 and 36 angles 282 us, this way 275,
// and 270 in plain sums), whole products in large tiles add runs of 64. The adjoint's error
// against 64 bits at that size is 2.1e-7 (2.9e-7 in plain sums, 1.9e-7 sample by sample), at 64^2
// x 32 and 12 angles 1.5e-7 (2.0e-7, 1.4e-7).
//
// Batches of products with few rows each (one per frequency or angle) take tiles of 64 columns
// whose height fits the rows: the least padding, a tile's loads of B counted as 24 rows. 127
// of 72 x 576 x 256 take 66 us in one tile of 72 rows each (20 TFMA/s), 74 us in two of 40, 90
// in three of 32 and 110 in two of 64. Where that leaves an SM without its three blocks, the
// smallest tiles: 72 of 64 x 288 x 256 in 23 us (25 us in tiles of 64 rows).
void launch_sgemm(const SgemmArgs *g, int n, cudaStream_t st) {
    constexpr int kWave = 3 * 152;
    int n64 = 0, n56 = 0, rows = 0;
    for (int i = 0; i < n; ++i) {
        n64 += sgemm_tiles(g[i]);
        n56 += (g[i].M + 55) / 56 * ((g[i].N + 127) / 128);
        if (g[i].nbatch != 1) rows = std::max(rows, g[i].M);
    }
    int height = 0;
    if (rows > 0) {
        for (int h : {32, 40, 56, 64, 72})
            if (!height || (rows + h - 1) / h * (h + 24) < (rows + height - 1) / height * (height + 24)) height = h;
        int64_t tiles = 0;
        for (int i = 0; i < n; ++i)
            tiles += (int64_t)g[i].nbatch * ((g[i].M + height - 1) / height) * ((g[i].N + 63) / 64);
        if (tiles < kWave) height = 32;
    }
    if (g[0].fine && g[0].half > 0) run<kFineRows, 128, 6, 8, 1>(g, n, st);
    else if (height == 40) run<40, 64, 5, 8, 2>(g, n, st);
    else if (height == 56) run<56, 64, 7, 8, 2>(g, n, st);
    else if (height == 64) run<64, 64, 8, 8, 2>(g, n, st);
    else if (height == 72) run<72, 64, 9, 8, 2>(g, n, st);
    else if (height == 0 && n64 >= 400 && (n56 + kWave - 1) / kWave * 56 < (n64 + kWave - 1) / kWave * 64)
        run<56, 128, 7, 8, 1>(g, n, st);
    else if (height == 0 && n64 >= 400) run<64, 128, 8, 8, 1>(g, n, st);
    else run<32, 64, 4, 8, 2>(g, n, st);
}

}  // namespace mpiffl
