// Tensor PSF: the line operator with coupled slices (Appendix B, Eq. (31)).
//
// An x drive read by a collinear coil takes h_uu(u, z) = 3 [L'(xi) u^2/rho^2 +
// (L(xi)/xi) z^2/rho^2], xi = rho / a, so the PSF-convolved projection of line l mixes every
// slice z: c_l = sum_z H_{l-z} b.p_z with H_d[e][i] = h_uu(u_lo + e/Q - i, d). Folded with
// the line operator W_par of the line's trajectory,
//     data[m][l] = g_m sum_z W_{par(l), l-z} (b . p)[m][z],    W_{par,d} = W_par H_d.
// H_d is even in d, so the sum over z is a product with a symmetric Toeplitz matrix, a corner
// of a symmetric circulant one of period L = 2 Nz, which the DFT along z makes diagonal with
// real values: with c_0 = c_Nz = 1 / L, c_f = 2 / L else, and
//     V_{par,f} = c_f W_par (H_0 + 2 sum_{0<d<Nz} H_d cos(2 pi f d / L)),
// the data are, over f = 0 .. Nz and both of cos and sin (sin(0) and sin(pi l) vanish),
//     data[m][l] = g_m sum_f t_f(l) V_{par(l),f} sum_z t_f(z) (b . p)[m][z],
// t_f(z) = cos(2 pi f z / L) or sin. That is 2 Nz products of one 2 n_b x N matrix and a
// vector per angle and trajectory, in the place of Nz^2 (of Nz^2 / 2 each with zig-zag).
//
// Three FP32 products (sgemm.cu) a direction: along z by t (2 Nz x Nz, one problem per angle),
// per frequency by V (rows: angles, cos and sin), and back along z (per trajectory: its
// lines). The rows q of a spectrum are cos 0, cos Nz, then cos and sin of f = 1 .. Nz - 1.
// Bound by the FP32 pipes: 2.0 GFMA a direction at 256^2 x 128 and 36 angles, 54 us at their
// rate, in 112 us forward and 116 us transposed (20 + 68 + 24 and 24 + 72 + 20). The same sum
// as one tensor-core product per line over all slices (87 GFLOP in three bf16 products) took
// 330 us a direction, with 12 times the error against 64 bits (5.5e-6 of the pair's outputs,
// 4.3e-7 this way).
#include <algorithm>
#include <cmath>
#include <vector>

#include "collapsed.h"
#include "fold.h"

namespace mpiffl {

namespace {

struct TenState {
    double fwhm = -1.0;     // of the tables; < 0: none
    int F = 0;              // frequencies, Nz + 1
    int Np = 0, Rp = 0;     // N and 2 n_b rounded up to 4: rows of 16-byte loads
    int ldt = 0, ldtp[2] = {0, 0};
    float *t = nullptr;     // [2 Nz][ldz] t_f(z), A of the step along z of the projections
    float *tp[2] = {nullptr, nullptr};  // [2 Nz][ldtp] its columns of each trajectory's lines
    float *tt = nullptr;    // [Nz][ldt] its transpose
    float *vf = nullptr;    // [F][N][n_par Rp] V transposed, B of the forward
    float *va = nullptr;    // [F][n_par Rp][Np] V, B of the adjoint
    int *rows = nullptr;    // 2 M spectrum rows of a frequency (angle, cos or sin), then M of one of them
    float *ps = nullptr;    // [M][2 Nz][Np] spectrum of the projections
    float *ds = nullptr;    // [M][2 Nz][n_par Rp] spectrum of the data
    float *pad = nullptr;   // input rows on 16 bytes, weighted by the coil map
    int ldz = 0;
};

TenState *ts(const mpi_ffl_handle *h) { return reinterpret_cast<TenState *>(h->ten_state); }

template <class T>
bool talloc(T **p, size_t n) {
    if (dev_malloc((void **)p, std::max<size_t>(1, n) * sizeof(T)) != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return false;
    }
    return true;
}

int up4(int n) { return (n + 3) / 4 * 4; }

// h_uu at in-plane offset (u, z) voxels; a = FWHM / (2 x_h)
double h_uu_host(double u, double z, double a) {
    const double rho2 = u * u + z * z;
    if (rho2 == 0.0) return 1.0;
    const double xi = std::sqrt(rho2) / a;
    double lx;  // L(xi) / xi
    if (xi < 0.05) {
        const double x2 = xi * xi;
        lx = 1.0 / 3.0 - x2 / 45.0 + 2.0 * x2 * x2 / 945.0 - x2 * x2 * x2 / 4725.0;
    } else {
        lx = (1.0 / std::tanh(xi) - 1.0 / xi) / xi;
    }
    return 3.0 * (langevin_d1_host(xi) * u * u / rho2 + lx * z * z / rho2);
}

// gf[f][k] = c_f (g[0][k] + 2 sum_{0<d<Nz} g[d][k] cos(2 pi f d / L)); cs[j] = cos(2 pi j / L)
__global__ void __launch_bounds__(256) k_ten_taps(const double *__restrict__ g, const double *__restrict__ cs,
                                                  double *__restrict__ gf, int Nz, int Lk) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x, f = blockIdx.y, L = 2 * Nz;
    if (k >= Lk) return;
    double acc = 0.0;
    int j = 0;
    for (int d = 1; d < Nz; ++d) {
        j += f;
        if (j >= L) j -= L;
        acc = fma(g[(size_t)d * Lk + k], cs[j], acc);
    }
    gf[(size_t)f * Lk + k] = (f == 0 || f == Nz ? 1.0 : 2.0) / L * (g[k] + 2.0 * acc);
}

// FP32 operands of V [n_par][F][R][N]: vf[f][i][par Rp + o] and va[f][par Rp + o][i], zero in
// the pads
__global__ void __launch_bounds__(256) k_ten_operands(const double *__restrict__ V, float *__restrict__ vf,
                                                      float *__restrict__ va, int n_par, int F, int R, int N, int Rp,
                                                      int Np) {
    const long long nr = (long long)n_par * Rp, total = F * nr * Np;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(t % Np), po = (int)(t / Np % nr), f = (int)(t / Np / nr);
        const int par = po / Rp, o = po % Rp;
        const float v = i < N && o < R ? (float)V[(((size_t)par * F + f) * R + o) * N + i] : 0.f;
        va[t] = v;
        if (i < N) vf[((size_t)f * N + i) * nr + po] = v;
    }
}

// V from W_par and the tensor PSF, in FP64 on the device, then its FP32 operands
bool build_v(mpi_ffl_handle *h, TenState *t) {
    const Dims &d = h->d;
    const int R = 2 * d.nb, kmin = fold_kmin(d), Lk = fold_taps(d), L = 2 * d.Nz;
    const double a = h->fwhm / (2.0 * langevin_half_point_host());
    std::vector<double> g((size_t)d.Nz * Lk), c(L);
    for (int dz = 0; dz < d.Nz; ++dz)
        for (int k = 0; k < Lk; ++k) g[(size_t)dz * Lk + k] = h_uu_host((double)(k + kmin) / d.Q, dz, a);
    for (int j = 0; j < L; ++j) c[j] = std::cos(2.0 * 3.14159265358979323846 * j / L);
    double *dg = nullptr, *dc = nullptr, *df = nullptr, *V = nullptr;
    bool ok = fold_w(h) == MPI_FFL_OK && talloc(&dg, g.size()) && talloc(&dc, c.size()) &&
              talloc(&df, (size_t)t->F * Lk) && talloc(&V, (size_t)d.n_par * t->F * R * d.N);
    if (ok) {
        cudaMemcpy(dg, g.data(), g.size() * sizeof(double), cudaMemcpyHostToDevice);
        cudaMemcpy(dc, c.data(), c.size() * sizeof(double), cudaMemcpyHostToDevice);
        k_ten_taps<<<dim3((Lk + 255) / 256, t->F), 256>>>(dg, dc, df, d.Nz, Lk);
        launch_fold_taps(fold_w_dev(h), df, V, d, d.n_par, t->F, nullptr);
        k_ten_operands<<<152 * 8, 256>>>(V, t->vf, t->va, d.n_par, t->F, R, d.N, t->Rp, t->Np);
        ok = cudaDeviceSynchronize() == cudaSuccess && cudaGetLastError() == cudaSuccess;
    }
    for (void *p : {(void *)dg, (void *)dc, (void *)df, (void *)V})
        if (p) dev_free(p);
    return ok;
}

bool build(mpi_ffl_handle *h, TenState *t) {
    const Dims &d = h->d;
    const int Q = 2 * d.Nz;
    t->F = d.Nz + 1;
    t->Np = up4(d.N);
    t->Rp = up4(2 * d.nb);
    t->ldz = up4(d.Nz);
    t->ldt = up4(Q);
    const size_t nr = (size_t)d.n_par * t->Rp, rows = (size_t)d.M * d.Nz;
    std::vector<float> T((size_t)Q * t->ldz, 0.f), Tt((size_t)d.Nz * t->ldt, 0.f);
    std::vector<double> c(4 * Q);  // two turns of cos in steps of pi / Q
    for (int j = 0; j < 4 * Q; ++j) c[j] = std::cos(3.14159265358979323846 * (j % (2 * Q)) / Q);
    for (int q = 0; q < Q; ++q)
        for (int z = 0; z < d.Nz; ++z) {
            const int f = q < 2 ? q * d.Nz : q / 2;
            // sin(x) = cos(x - pi / 2), Q / 2 steps of the table
            const int j = (int)(2LL * f * z % (2 * Q));
            const float v = (float)(q >= 2 && q % 2 ? c[j + 2 * Q - Q / 2] : c[j]);
            T[(size_t)q * t->ldz + z] = v;
            Tt[(size_t)z * t->ldt + q] = v;
        }
    std::vector<int> idx;
    for (int m = 0; m < d.M; ++m)
        for (int part = 0; part < 2; ++part) idx.push_back(m * Q + part);
    for (int m = 0; m < d.M; ++m) idx.push_back(m * Q);
    bool ok = talloc(&t->t, T.size()) && talloc(&t->tt, Tt.size()) && talloc(&t->rows, idx.size()) &&
              talloc(&t->vf, (size_t)t->F * d.N * nr) && talloc(&t->va, (size_t)t->F * nr * t->Np) &&
              talloc(&t->ps, (size_t)d.M * Q * t->Np) && talloc(&t->ds, (size_t)d.M * Q * nr) &&
              talloc(&t->pad, rows * std::max(t->Np, t->Rp));
    for (int par = 0; ok && par < d.n_par; ++par) {
        const int n = (d.Nz - par + d.n_par - 1) / d.n_par;
        t->ldtp[par] = std::max(4, up4(n));
        std::vector<float> Tp((size_t)Q * t->ldtp[par], 0.f);
        for (int q = 0; q < Q; ++q)
            for (int l = 0; l < n; ++l)
                Tp[(size_t)q * t->ldtp[par] + l] = T[(size_t)q * t->ldz + par + l * d.n_par];
        ok = talloc(&t->tp[par], Tp.size()) &&
             cudaMemcpy(t->tp[par], Tp.data(), Tp.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess;
    }
    ok = ok && cudaMemcpy(t->t, T.data(), T.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(t->tt, Tt.data(), Tt.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(t->rows, idx.data(), idx.size() * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess;
    return ok && build_v(h, t);
}

// One problem of a batch; the rest of the fields are zero.
SgemmArgs product(const float *A, int64_t lda, int M, int K, const float *B, int ldb, int bcols, float *C, int64_t ldc,
                  int N, int nbatch, int64_t sA, int64_t sB, int64_t sC) {
    SgemmArgs g{};
    g.A = A;
    g.lda = lda;
    g.M = M;
    g.K = K;
    g.B = B;
    g.ldb = ldb;
    g.bcols = bcols;
    g.C = C;
    g.ldc = ldc;
    g.N = N;
    g.rdiv = 1;
    g.nbatch = nbatch;
    g.sA = sA;
    g.sB = sB;
    g.sC = sC;
    return g;
}

// The products by V: in [M][2 Nz][ldi] -> out [M][2 Nz][ldo] with B [F][K][ldb], K values of
// in, N of out, gain per angle.
void per_frequency(const mpi_ffl_handle *h, const TenState *t, const float *in, int ldi, int K, const float *B, int ldb,
                   float *out, int ldo, int N, cudaStream_t st) {
    const Dims &d = h->d;
    const int64_t per = (int64_t)K * ldb;
    SgemmArgs g[3];
    // f = 1 .. Nz - 1: rows (angle, cos or sin) from spectrum row 2 f on; then f = 0 and Nz
    g[0] = product(in + 2 * ldi, ldi, 2 * d.M, K, B + per, ldb, ldb, out + 2 * ldo, ldo, N, d.Nz - 1, 2 * ldi, per,
                   2 * ldo);
    g[1] = product(in, ldi, d.M, K, B, ldb, ldb, out, ldo, N, 1, 0, 0, 0);
    g[2] = product(in + ldi, ldi, d.M, K, B + per * d.Nz, ldb, ldb, out + ldo, ldo, N, 1, 0, 0, 0);
    for (int i = 0; i < 3; ++i) {
        g[i].arow = g[i].crow = t->rows + (i ? 2 * d.M : 0);
        g[i].scale = h->t_gain;
        g[i].rdiv = 2 * d.Nz;
    }
    launch_sgemm(g, 3, st);
}

}  // namespace

int ten_init(mpi_ffl_handle *h) {
    if (!col_supported(h)) return MPI_FFL_ERR_UNSUPPORTED;
    TenState *t = ts(h);
    if (!t) h->ten_state = t = new TenState();
    t->fwhm = -1.0;
    if (!(t->vf ? build_v(h, t) : build(h, t))) {
        ten_release(h);
        cudaGetLastError();
        return MPI_FFL_ERR_OOM;
    }
    t->fwhm = h->fwhm;
    return MPI_FFL_OK;
}

bool ten_ready(const mpi_ffl_handle *h) { return ts(h) && ts(h)->fwhm == h->fwhm; }

BufferList ten_buffers(const mpi_ffl_handle *h) {
    const TenState *t = ts(h);
    if (!t) return {};
    return {t->t, t->tp[0], t->tp[1], t->tt, t->vf, t->va, t->rows, t->ps, t->ds, t->pad};
}

void ten_release(mpi_ffl_handle *h) {
    TenState *t = ts(h);
    if (!t) return;
    for (void *p : ten_buffers(h)) dev_free(p);
    delete t;
    h->ten_state = nullptr;
}

void ten_forward(mpi_ffl_handle *h, const float *proj, const float *coil, float *data, cudaStream_t st) {
    const Dims &d = h->d;
    const TenState *t = ts(h);
    const int R = 2 * d.nb, Q = 2 * d.Nz, nr = d.n_par * t->Rp;
    int ldp = d.N;
    if (coil || d.N % 4 || (reinterpret_cast<uintptr_t>(proj) & 15)) {
        launch_coil_pad(proj, coil, t->pad, (long long)d.M * d.Nz, d.Nz, d.N, t->Np, st);
        h->launches++;
        proj = t->pad;
        ldp = t->Np;
    }
    const SgemmArgs z = product(t->t, t->ldz, Q, d.Nz, proj, ldp, ldp, t->ps, t->Np, d.N, d.M, 0, (int64_t)d.Nz * ldp,
                                (int64_t)Q * t->Np);
    launch_sgemm(&z, 1, st);
    per_frequency(h, t, t->ps, t->Np, d.N, t->vf, nr, t->ds, nr, nr, st);
    SgemmArgs g[2];
    for (int par = 0; par < d.n_par; ++par)
        g[par] = product(t->tt + (size_t)par * t->ldt, (int64_t)d.n_par * t->ldt,
                         (d.Nz - par + d.n_par - 1) / d.n_par, Q, t->ds + par * t->Rp, nr, t->Rp,
                         data + (size_t)par * R, (int64_t)d.n_par * R, R, d.M, 0, (int64_t)Q * nr, (int64_t)d.Nz * R);
    launch_sgemm(g, d.n_par, st);
    h->launches += 2;  // three products in the caller's timed stage
}

void ten_adjoint(mpi_ffl_handle *h, const float *data, const float *coil, float *proj, cudaStream_t st) {
    const Dims &d = h->d;
    const TenState *t = ts(h);
    const int R = 2 * d.nb, Q = 2 * d.Nz, nr = d.n_par * t->Rp;
    if (R % 4 || (reinterpret_cast<uintptr_t>(data) & 15)) {
        launch_coil_pad(data, nullptr, t->pad, (long long)d.M * d.Nz, d.Nz, R, t->Rp, st);
        h->launches++;
        data = t->pad;
    }
    SgemmArgs g[2];
    for (int par = 0; par < d.n_par; ++par)
        g[par] = product(t->tp[par], t->ldtp[par], Q, (d.Nz - par + d.n_par - 1) / d.n_par, data + (size_t)par * t->Rp,
                         d.n_par * t->Rp, t->Rp, t->ds + par * t->Rp, nr, t->Rp, d.M, 0, (int64_t)d.Nz * t->Rp,
                         (int64_t)Q * nr);
    launch_sgemm(g, d.n_par, st);
    per_frequency(h, t, t->ds, nr, nr, t->va, t->Np, t->ps, t->Np, d.N, st);
    const SgemmArgs z = product(t->tt, t->ldt, d.Nz, Q, t->ps, t->Np, t->Np, proj, d.N, d.N, d.M, 0,
                                (int64_t)Q * t->Np, (int64_t)d.Nz * d.N);
    launch_sgemm(&z, 1, st);
    h->launches += 2;
    if (coil) {
        launch_coil_pad(proj, coil, proj, (long long)d.M * d.Nz, d.Nz, d.N, d.N, st);
        h->launches++;
    }
}

}  // namespace mpiffl
