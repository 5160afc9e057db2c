// Solver kernels for Eq. (26) (Sec. 3.3) and the FP64 reductions it needs.
//
// Reductions are deterministic: each block writes one FP64 partial sum in a fixed
// order and a single block adds the partials in index order (in the solve and the power
// iteration the last block to finish, in the same launch).
// The stop test leaves its verdict in a device flag; the host reads it only when
// an early stop was requested. The optional `done` flag of the per-iteration
// kernels turns them into no-ops once it is set.
#include <algorithm>
#include <initializer_list>

#include "internal.h"
#include "tc_ptx.cuh"

namespace mpiffl {

constexpr int kRedThreads = 256;

int reduce_blocks(int64_t n) {
    int64_t b = (n + kRedThreads * 4 - 1) / (kRedThreads * 4);
    if (b > 1024) b = 1024;
    if (b < 1) b = 1;
    return (int)b;
}

__device__ __forceinline__ double block_sum(double v) {
    __shared__ double sh[kRedThreads / 32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
    __syncthreads();
    return t;  // valid in thread 0
}

// True in every thread of the last block of the launch to arrive, with the other blocks'
// partials visible; *counter is left at 0 for the next launch.
__device__ __forceinline__ bool last_block(unsigned *counter) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
        if (last) *counter = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

__device__ __forceinline__ double sum_partials(const double *partials, int n) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc += __ldcg(partials + i);
    return block_sum(acc);
}

// 16-byte accesses when every pointer is on 16 bytes
inline bool vec4(std::initializer_list<const void *> p) {
    for (const void *q : p)
        if (reinterpret_cast<uintptr_t>(q) & 15) return false;
    return true;
}

template <bool VEC>
__global__ void __launch_bounds__(256) k_momentum(const float *__restrict__ x, const float *__restrict__ xp,
                                                  float *__restrict__ y, float beta, int64_t n, const int *done) {
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    if (done && *done) return;
    const int64_t step = (int64_t)gridDim.x * blockDim.x, i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    auto f = [beta](float xi, float pi) { return fmaf(beta, xi - pi, xi); };
    if (VEC)
        for (int64_t i = i0; i < n / 4; i += step) {
            const float4 a = reinterpret_cast<const float4 *>(x)[i], b = reinterpret_cast<const float4 *>(xp)[i];
            reinterpret_cast<float4 *>(y)[i] = make_float4(f(a.x, b.x), f(a.y, b.y), f(a.z, b.z), f(a.w, b.w));
        }
    for (int64_t i = (VEC ? n / 4 * 4 : 0) + i0; i < n; i += step) y[i] = f(x[i], xp[i]);
}

void launch_momentum(const float *x, const float *xp, float *y, double beta_num, int64_t n, const int *done,
                     cudaStream_t st) {
    const bool v = vec4({x, xp, y});
    const int blocks = (int)std::min<int64_t>((n / (v ? 4 : 1) + 255) / 256 + 1, 152 * 8);
    launch_dependent(v ? k_momentum<true> : k_momentum<false>, dim3(blocks), dim3(256), 0, st, x, xp, y,
                     (float)beta_num, n, done);
}

// One launch per iteration for r <- r - b, hist[k] = ||r|| (FP64) and the stop test: *stop
// is set when the relative change from hist[k-1] is at most stop_rel (1) or the norm is not
// finite (2), and *iters_done counts the iterations whose test ran. With the sum and the test
// in two further launches of one block this took 12 us at 128^2 x 64 (24 angles), now 9 us.
template <bool VEC>
__global__ void __launch_bounds__(kRedThreads) k_residual(float *__restrict__ r, const float *__restrict__ b,
                                                          int64_t n, double *partials, unsigned *counter,
                                                          double *hist, int k, double stop_rel, int *stop,
                                                          int *iters_done, const int *frozen) {
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    if (frozen && *frozen) return;  // the whole launch
    double acc = 0.0;
    const int64_t step = (int64_t)gridDim.x * blockDim.x, i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (VEC)
        for (int64_t i = i0; i < n / 4; i += step) {
            const float4 p = reinterpret_cast<const float4 *>(r)[i], q = reinterpret_cast<const float4 *>(b)[i];
            const float4 v = make_float4(p.x - q.x, p.y - q.y, p.z - q.z, p.w - q.w);
            reinterpret_cast<float4 *>(r)[i] = v;
            acc += (double)v.x * (double)v.x + (double)v.y * (double)v.y + (double)v.z * (double)v.z +
                   (double)v.w * (double)v.w;
        }
    for (int64_t i = (VEC ? n / 4 * 4 : 0) + i0; i < n; i += step) {
        const float v = r[i] - b[i];
        r[i] = v;
        acc += (double)v * (double)v;
    }
    const double t = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = t;
    if (!last_block(counter)) return;
    const double sq = sum_partials(partials, gridDim.x);
    if (threadIdx.x != 0 || *stop) return;
    const double norm = sqrt(sq);
    hist[k] = norm;
    *iters_done = k + 1;
    if (!(norm == norm) || norm > 1e300) {
        *stop = 2;
    } else if (stop_rel > 0.0 && k > 0) {
        const double prev = hist[k - 1];
        if (fabs(prev - norm) <= stop_rel * prev) *stop = 1;
    }
}

void launch_residual(float *r, const float *b, int64_t n, double *partials, unsigned *counter, double *hist, int k,
                     double stop_rel, int *stop, int *iters_done, const int *frozen, cudaStream_t st) {
    const bool v = vec4({r, b});
    const int blocks = (int)std::min<int64_t>(std::max<int64_t>(1, (n + 2047) / 2048), 152 * 4);
    launch_dependent(v ? k_residual<true> : k_residual<false>, dim3(blocks), dim3(kRedThreads), 0, st, r, b, n,
                     partials, counter, hist, k, stop_rel, stop, iters_done, frozen);
}

// The power iteration's inner products in one pass: *ww = <w, w>, *scale = 1 / sqrt(<w, w>),
// which k_scale applies, and with BOTH (the last step, whose Rayleigh quotient is the
// result) *vw = <v, w>. Bound by the FP64 pipe: a conversion and an FMA an element cost more
// than its read. (Two products, two sums of partials and a scaling with a square root per
// thread took 54 us a step at 128^2 x 64, now 16 us.)
template <bool VEC, bool BOTH>
__global__ void __launch_bounds__(kRedThreads) k_dot2(const float *__restrict__ v, const float *__restrict__ w,
                                                      int64_t n, double *partials, unsigned *counter, double *vw,
                                                      double *ww, float *scale) {
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    double a[4] = {0.0, 0.0, 0.0, 0.0}, b[4] = {0.0, 0.0, 0.0, 0.0};
    const int64_t step = (int64_t)gridDim.x * blockDim.x, i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    auto add = [&](int u, float x, float y) {
        const double yd = y;
        if (BOTH) a[u] = fma((double)x, yd, a[u]);
        b[u] = fma(yd, yd, b[u]);
    };
    if (VEC)
#pragma unroll 2
        for (int64_t i = i0; i < n / 4; i += step) {
            const float4 q = reinterpret_cast<const float4 *>(w)[i];
            const float4 p = BOTH ? reinterpret_cast<const float4 *>(v)[i] : q;
            add(0, p.x, q.x);
            add(1, p.y, q.y);
            add(2, p.z, q.z);
            add(3, p.w, q.w);
        }
    for (int64_t i = (VEC ? n / 4 * 4 : 0) + i0; i < n; i += step) add(0, BOTH ? v[i] : 0.f, w[i]);
    const double tb = block_sum((b[0] + b[1]) + (b[2] + b[3]));
    double ta = 0.0;
    if (BOTH) ta = block_sum((a[0] + a[1]) + (a[2] + a[3]));
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = tb;
        if (BOTH) partials[gridDim.x + blockIdx.x] = ta;
    }
    if (!last_block(counter)) return;
    const double sb = sum_partials(partials, gridDim.x);
    double sa = 0.0;
    if (BOTH) sa = sum_partials(partials + gridDim.x, gridDim.x);
    if (threadIdx.x == 0) {
        if (BOTH) *vw = sa;
        *ww = sb;
        *scale = sb > 0.0 ? (float)(1.0 / sqrt(sb)) : 0.f;
    }
}

int dot2_blocks(int64_t n) { return (int)std::min<int64_t>(std::max<int64_t>(1, (n + 2047) / 2048), 152 * 2); }

void launch_dot2(const float *v, const float *w, int64_t n, double *partials, unsigned *counter, double *vw,
                 double *ww, float *scale, cudaStream_t st) {
    const bool a = vec4({v, w});
    auto kernel = vw ? (a ? k_dot2<true, true> : k_dot2<false, true>) : (a ? k_dot2<true, false> : k_dot2<false, false>);
    launch_dependent(kernel, dim3(dot2_blocks(n)), dim3(kRedThreads), 0, st, v, w, n, partials, counter, vw, ww,
                     scale);
}

__global__ void __launch_bounds__(kRedThreads) k_dot(const float *__restrict__ a, const float *__restrict__ b,
                                                     int64_t n, double *partials) {
    double acc = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        acc += (double)a[i] * (double)b[i];
    const double t = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

void launch_dot(const float *a, const float *b, int64_t n, double *partials, int nblk, cudaStream_t st) {
    k_dot<<<nblk, kRedThreads, 0, st>>>(a, b, n, partials);
}

__global__ void __launch_bounds__(kRedThreads) k_finalize(const double *partials, int nblk, double *out) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) acc += partials[i];
    const double t = block_sum(acc);
    if (threadIdx.x == 0) *out = t;
}

void launch_finalize(const double *partials, int nblk, double *out, cudaStream_t st) {
    k_finalize<<<1, kRedThreads, 0, st>>>(partials, nblk, out);
}

__global__ void __launch_bounds__(kRedThreads) k_finalize_f(const double *partials, int nblk, float *out) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) acc += partials[i];
    const double t = block_sum(acc);
    if (threadIdx.x == 0) *out = (float)t;
}

void launch_finalize_to_float(const double *partials, int nblk, float *out, cudaStream_t st) {
    k_finalize_f<<<1, kRedThreads, 0, st>>>(partials, nblk, out);
}

// Per-angle dot products: blockIdx.y = angle, per_angle contiguous floats each.
__global__ void __launch_bounds__(kRedThreads) k_angle_dots(const float *__restrict__ a, const float *__restrict__ b,
                                                            int64_t per_angle, double *partials) {
    const float *pa = a + (size_t)blockIdx.y * per_angle;
    const float *pb = b + (size_t)blockIdx.y * per_angle;
    double acc = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < per_angle; i += (int64_t)gridDim.x * blockDim.x)
        acc += (double)pa[i] * (double)pb[i];
    const double t = block_sum(acc);
    if (threadIdx.x == 0) partials[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = t;
}

void launch_angle_dots(const float *a, const float *b, int M, int64_t per_angle, double *partials,
                       int nblk_per_angle, cudaStream_t st) {
    dim3 grid(nblk_per_angle, M);
    k_angle_dots<<<grid, kRedThreads, 0, st>>>(a, b, per_angle, partials);
}

__global__ void __launch_bounds__(kRedThreads) k_angle_finalize(const double *partials, int nblk, float *out) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) acc += partials[(size_t)blockIdx.x * nblk + i];
    const double t = block_sum(acc);
    if (threadIdx.x == 0) out[blockIdx.x] = (float)t;
}

void launch_angle_finalize(const double *partials, int M, int nblk_per_angle, float *out, cudaStream_t st) {
    k_angle_finalize<<<M, kRedThreads, 0, st>>>(partials, nblk_per_angle, out);
}

// partials are [angle][nblk]: each angle's sum weighted, in one sum over threads in a fixed order
__global__ void __launch_bounds__(kRedThreads) k_angles_weighted(const double *partials, int M, int nblk,
                                                                 const float *__restrict__ weight, float *out) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < M * nblk; i += blockDim.x) acc += (double)__ldg(weight + i / nblk) * partials[i];
    const double t = block_sum(acc);
    if (threadIdx.x == 0) *out = (float)t;
}

void launch_angles_weighted(const double *partials, int M, int nblk_per_angle, const float *weight, float *out,
                            cudaStream_t st) {
    k_angles_weighted<<<1, kRedThreads, 0, st>>>(partials, M, nblk_per_angle, weight, out);
}

// T^T T x with forward differences and no wrap (Neumann): 7-point stencil with the
// face-reduced diagonal.
__device__ __forceinline__ float ttt_at(const float *__restrict__ x, int N, int Nz, int z, int y, int xx) {
    const size_t i = ((size_t)z * N + y) * N + xx;
    const float c = x[i];
    float s = 0.f;
    if (xx > 0) s += c - x[i - 1];
    if (xx < N - 1) s += c - x[i + 1];
    if (y > 0) s += c - x[i - N];
    if (y < N - 1) s += c - x[i + N];
    if (z > 0) s += c - x[i - (size_t)N * N];
    if (z < Nz - 1) s += c - x[i + (size_t)N * N];
    return s;
}

__global__ void k_ttt(const float *__restrict__ x, float *__restrict__ out, int N, int Nz) {
    const int xx = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, z = blockIdx.z;
    if (xx >= N) return;
    out[((size_t)z * N + y) * N + xx] = ttt_at(x, N, Nz, z, y, xx);
}

void launch_ttt(const float *x, float *out, int N, int Nz, cudaStream_t st) {
    dim3 grid((N + 127) / 128, N, Nz);
    k_ttt<<<grid, 128, 0, st>>>(x, out, N, Nz);
}

// x_out = P(y - tau (g + lam T^T T y)), P = max(0, .) when nonneg. Once *done is set
// the solve is frozen: x_out = xcur (the current iterate), so that the buffer swap of
// the next iteration keeps the final iterate. VEC: four voxels of a row a thread (N % 4 ==
// 0, pointers on 16 bytes); the terms of T^T T are added in ttt_at's order.
template <bool VEC>
__device__ __forceinline__ void update_row(const float *__restrict__ y, const float *__restrict__ g,
                                           float *__restrict__ xo, float tau, float lam, int nonneg, int N, int Nz,
                                           bool frozen, const float *__restrict__ xcur, int row) {
    constexpr int V = VEC ? 4 : 1;
    const int yy = row % N, z = row / N;
    for (int xx = V * (threadIdx.x & 31); xx < N; xx += V * 32) {
        const size_t i = ((size_t)z * N + yy) * N + xx;
        if (frozen) {
            if (xcur)
#pragma unroll
                for (int u = 0; u < V; ++u) xo[i + u] = xcur[i + u];
            continue;
        }
        if (VEC) {
            auto at = [&](size_t k) { return *reinterpret_cast<const float4 *>(y + k); };
            const size_t sl = (size_t)N * N;
            const float4 c4 = at(i), g4 = *reinterpret_cast<const float4 *>(g + i);
            const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 ym = yy > 0 ? at(i - N) : z4, yp = yy < N - 1 ? at(i + N) : z4;
            const float4 zm = z > 0 ? at(i - sl) : z4, zp = z < Nz - 1 ? at(i + sl) : z4;
            const float left = xx > 0 ? y[i - 1] : 0.f, right = xx + 4 < N ? y[i + 4] : 0.f;
            const float c[6] = {left, c4.x, c4.y, c4.z, c4.w, right};
            const float gv[4] = {g4.x, g4.y, g4.z, g4.w};
            const float a0[4] = {ym.x, ym.y, ym.z, ym.w}, a1[4] = {yp.x, yp.y, yp.z, yp.w};
            const float b0[4] = {zm.x, zm.y, zm.z, zm.w}, b1[4] = {zp.x, zp.y, zp.z, zp.w};
            float o[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float cc = c[u + 1];
                float s = 0.f;
                if (xx + u > 0) s += cc - c[u];
                if (xx + u < N - 1) s += cc - c[u + 2];
                if (yy > 0) s += cc - a0[u];
                if (yy < N - 1) s += cc - a1[u];
                if (z > 0) s += cc - b0[u];
                if (z < Nz - 1) s += cc - b1[u];
                const float v = fmaf(-tau, fmaf(lam, s, gv[u]), cc);
                o[u] = nonneg ? fmaxf(v, 0.f) : v;
            }
            *reinterpret_cast<float4 *>(xo + i) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
            const float grad = fmaf(lam, ttt_at(y, N, Nz, z, yy, xx), g[i]);
            float v = fmaf(-tau, grad, y[i]);
            if (nonneg) v = fmaxf(v, 0.f);
            xo[i] = v;
        }
    }
}

// a warp per row (z, y)
template <bool VEC>
__global__ void __launch_bounds__(128) k_update(const float *__restrict__ y, const float *__restrict__ g,
                                                float *__restrict__ xo, float tau, float lam, int nonneg, int N,
                                                int Nz, const int *done, const float *__restrict__ xcur) {
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    const int row = blockIdx.x * 4 + threadIdx.x / 32;
    if (row < N * Nz) update_row<VEC>(y, g, xo, tau, lam, nonneg, N, Nz, done && *done, xcur, row);
}

void launch_update(const float *y, const float *g, float *xout, float tau, float lam, int nonneg,
                   int N, int Nz, const int *done, cudaStream_t st, const float *xcur) {
    const bool v = N % 4 == 0 && vec4({y, g, xout});
    launch_dependent(v ? k_update<true> : k_update<false>, dim3((N * Nz + 3) / 4), dim3(128), 0, st, y, g, xout, tau,
                     lam, nonneg, N, Nz, done, xcur);
}

// Per kept bin q: sum over segments of |b[seg][q]|^2 in FP64, segments in order.
__global__ void k_bin_energy(const float2 *__restrict__ data, int nseg, int nb, double *__restrict__ out) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nb) return;
    double acc = 0.0;
    for (int sgi = 0; sgi < nseg; ++sgi) {
        const float2 v = data[(size_t)sgi * nb + q];
        acc = fma((double)v.x, (double)v.x, fma((double)v.y, (double)v.y, acc));
    }
    out[q] = acc;
}

void launch_bin_energy(const float *data, int nseg, int nb, double *out, cudaStream_t st) {
    k_bin_energy<<<(nb + 127) / 128, 128, 0, st>>>(reinterpret_cast<const float2 *>(data), nseg, nb, out);
}

// frozen = stop (after the update of the stopping iteration)
__global__ void k_freeze(const int *stop, int *frozen) {
    if (*stop) *frozen = 1;
}

void launch_freeze(const int *stop, int *frozen, cudaStream_t st) { k_freeze<<<1, 1, 0, st>>>(stop, frozen); }

// SplitMix64 (Steele, Lea, Flood 2014) evaluated at counter i + 1: u in [-1, 1).
__global__ void k_splitmix_fill(float *v, int64_t n, uint64_t seed) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t z = seed + (uint64_t)(i + 1) * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        v[i] = (float)((double)(z >> 11) * 0x1.0p-52 - 1.0);
    }
}

void launch_splitmix_fill(float *v, int64_t n, uint64_t seed, cudaStream_t st) {
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, 152 * 16);
    k_splitmix_fill<<<blocks, 256, 0, st>>>(v, n, seed);
}

// out = *scale in
template <bool VEC>
__global__ void __launch_bounds__(256) k_scale(const float *in, float *out, int64_t n, const float *scale) {
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    const float s = *scale;
    const int64_t step = (int64_t)gridDim.x * blockDim.x, i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (VEC)
        for (int64_t i = i0; i < n / 4; i += step) {
            const float4 a = reinterpret_cast<const float4 *>(in)[i];
            reinterpret_cast<float4 *>(out)[i] = make_float4(a.x * s, a.y * s, a.z * s, a.w * s);
        }
    for (int64_t i = (VEC ? n / 4 * 4 : 0) + i0; i < n; i += step) out[i] = in[i] * s;
}

void launch_scale(const float *in, float *out, int64_t n, const float *scale, cudaStream_t st) {
    const bool v = vec4({in, out});
    const int blocks = (int)std::min<int64_t>((n / (v ? 4 : 1) + 255) / 256 + 1, 152 * 8);
    launch_dependent(v ? k_scale<true> : k_scale<false>, dim3(blocks), dim3(256), 0, st, in, out, n, scale);
}

// ---------------------------------------------------------------------- batches
__device__ __forceinline__ int batch_find_s(const int *__restrict__ offs, int n, int b) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(offs + mid) <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

constexpr int kVecPerBlock = 256 * 8;  // elements per block of the batched element-wise kernels

// The batched kernels are persistent: a grid of at most as many blocks as the GPU holds
// at once loops over the work items (item b belongs to the job j with offs[j] <= b <
// offs[j + 1]), so one launch per kind serves every job whatever their count and sizes.
// An item's arithmetic does not depend on the block that runs it.
__global__ void __launch_bounds__(256) k_momentum_batch(const MomentumJob *__restrict__ jobs,
                                                        const int *__restrict__ offs, int n, int total) {
    for (int bi = blockIdx.x; bi < total; bi += gridDim.x) {
        const int j = batch_find_s(offs, n, bi);
        const MomentumJob J = jobs[j];
        if (J.done && *J.done) continue;
        const int64_t base = (int64_t)(bi - offs[j]) * kVecPerBlock;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t i = base + u * 256 + threadIdx.x;
            if (i < J.n) {
                const float xi = J.x[i];
                J.y[i] = fmaf(J.beta, xi - J.xp[i], xi);
            }
        }
    }
}

__global__ void __launch_bounds__(kRedThreads) k_residual_batch(const ResidualJob *__restrict__ jobs,
                                                                const int *__restrict__ offs, int n, int total) {
    for (int bi = blockIdx.x; bi < total; bi += gridDim.x) {
        const int j = batch_find_s(offs, n, bi);
        const ResidualJob J = jobs[j];
        if (J.done && *J.done) continue;  // uniform over the block
        const int b = bi - offs[j];
        double acc = 0.0;
        for (int64_t i = (int64_t)b * blockDim.x + threadIdx.x; i < J.n; i += (int64_t)J.nblk * blockDim.x) {
            const float v = J.r[i] - J.b[i];
            J.r[i] = v;
            acc += (double)v * (double)v;
        }
        const double t = block_sum(acc);
        if (threadIdx.x == 0) J.partials[b] = t;
        __syncthreads();  // block_sum's shared words are reused by the next item
    }
}

// one block per problem: partial sums in index order, then the stop test
__global__ void __launch_bounds__(kRedThreads) k_stop_batch(const StopJob *__restrict__ jobs, int n) {
    for (int bi = blockIdx.x; bi < n; bi += gridDim.x) {
        const StopJob J = jobs[bi];
        if (*J.done) continue;
        double acc = 0.0;
        for (int i = threadIdx.x; i < J.nblk; i += blockDim.x) acc += J.partials[i];
        const double t = block_sum(acc);
        if (threadIdx.x == 0) {
            const double r = sqrt(t);
            J.hist[J.k] = r;
            J.flags[1] = J.k + 1;
            if (!(r == r) || r > 1e300) {
                J.flags[0] = 2;
            } else if (J.stop_rel > 0.0 && J.k > 0) {
                const double prev = J.hist[J.k - 1];
                if (fabs(prev - r) <= J.stop_rel * prev) J.flags[0] = 1;
            }
        }
        __syncthreads();
    }
}

// a frozen job keeps the final iterate in the buffer that becomes x
__global__ void __launch_bounds__(128) k_update_batch(const UpdateJob *__restrict__ jobs, const int *__restrict__ offs,
                                                      int n, int total) {
    for (int bi = blockIdx.x; bi < total; bi += gridDim.x) {
        const int j = batch_find_s(offs, n, bi);
        const UpdateJob J = jobs[j];
        const bool frozen = J.done && *J.done;
        for (int q = 0; q < 2; ++q) {
            const int row = (bi - offs[j]) * 8 + 4 * q + threadIdx.x / 32;
            if (row >= J.N * J.Nz) break;
            if (J.vec) update_row<true>(J.y, J.g, J.xo, J.tau, J.lam, J.nonneg, J.N, J.Nz, frozen, J.xcur, row);
            else update_row<false>(J.y, J.g, J.xo, J.tau, J.lam, J.nonneg, J.N, J.Nz, frozen, J.xcur, row);
        }
    }
}

int update_blocks(int N, int Nz) { return (N * Nz + 7) / 8; }

__global__ void k_freeze_batch(const StopJob *__restrict__ jobs, int n) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n && jobs[j].flags[0] != 0) *jobs[j].done = 1;
}

void launch_freeze_batch(const StopJob *jobs, int n, cudaStream_t st) {
    k_freeze_batch<<<(n + 127) / 128, 128, 0, st>>>(jobs, n);
}

// Blocks of a persistent batched launch: what the GPU holds at once, at most one per item.
template <class K>
int persistent_grid(K kernel, int threads, size_t smem, int total) {
    static int n_sm = 0;
    if (!n_sm) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        if (n_sm <= 0) n_sm = 1;
    }
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess || per < 1) {
        (void)cudaGetLastError();  // a failed query is not the caller's error
        per = 1;
    }
    return std::max(1, std::min(total, per * n_sm));
}

void launch_momentum_batch(const MomentumJob *jobs, const int *offs, int n, int total, cudaStream_t st) {
    if (total <= 0) return;
    k_momentum_batch<<<persistent_grid(k_momentum_batch, 256, 0, total), 256, 0, st>>>(jobs, offs, n, total);
}
void launch_residual_batch(const ResidualJob *jobs, const int *offs, int n, int total, cudaStream_t st) {
    if (total <= 0) return;
    k_residual_batch<<<persistent_grid(k_residual_batch, kRedThreads, 0, total), kRedThreads, 0, st>>>(jobs, offs, n,
                                                                                                       total);
}
void launch_stop_batch(const StopJob *jobs, int n, cudaStream_t st) {
    if (n <= 0) return;
    k_stop_batch<<<persistent_grid(k_stop_batch, kRedThreads, 0, n), kRedThreads, 0, st>>>(jobs, n);
}
void launch_update_batch(const UpdateJob *jobs, const int *offs, int n, int total, cudaStream_t st) {
    if (total <= 0) return;
    k_update_batch<<<persistent_grid(k_update_batch, 128, 0, total), 128, 0, st>>>(jobs, offs, n, total);
}

}  // namespace mpiffl
