// The line operator of one trajectory folded to one matrix (Sec. 2.1, Eq. (13)).
//
// Every raster line of a trajectory (line parity) sees the same E, V and band DFT, so
// W = S D_Gamma F V E is one matrix per trajectory and W H, with the PSF folded in, takes
// a projection straight to the line's kept bins:
//     W[o][e] = D_o L^-1/2 sum_j e^{2 pi i w_o j / L} (w0_j [n_j = e] + w1_j [n_j + 1 = e])
//     data[line] = g_m (W H) proj[line],   proj[line] = g_m (W H)^T data[line]
// Both are built here in FP64 on the device; the tensor-core paths split them to hi + lo
// operands (collapsed.cu), the staged path applies W H in FP32 (sgemm.cu).
#include <cmath>
#include <vector>

#include "collapsed.h"
#include "fold.h"

namespace mpiffl {

namespace {

struct FoldState {
    double *W = nullptr;     // [n_par][2 n_b][N_e]
    double *taps = nullptr;  // PSF taps of slot 0, then of slot 1
    double taps_fwhm = -1.0; // their width; < 0: none
    double *WH = nullptr;    // [n_par][slots folded together][2 n_b][N]
    // FP32 operands: B of the forward [n_par][N][ldf] of slot 0 (h) and 1 (d h / d fwhm), and of
    // the adjoint [n_par][2 n_b][lda] of slot 0
    float *f[2] = {nullptr, nullptr}, *a = nullptr;
    bool used[2] = {false, false};   // a call has applied the slot
    bool ready[2] = {false, false};  // its operands are those of the handle's width
    int ldf = 0, lda = 0;
    int *rows = nullptr;  // lines of trajectory 0, then of trajectory 1
    int nrows[2] = {0, 0};
};

FoldState *fs(const mpi_ffl_handle *h) { return reinterpret_cast<FoldState *>(h->fold_state); }

// Host data to device memory, there when this returns: a copy from pageable memory may return
// before, on the legacy stream, which the caller's non-blocking stream does not wait for.
template <class T>
bool fupload(T *p, const std::vector<T> &v) {
    return cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) == cudaSuccess &&
           cudaStreamSynchronize(nullptr) == cudaSuccess;
}

template <class T>
bool falloc(T **p, size_t n) {
    if (*p) return true;
    if (dev_malloc((void **)p, n * sizeof(T)) != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return false;
    }
    return true;
}

// A block owns one fine cell of one trajectory, a thread one kept bin: the samples that
// touch the cell (its CSR list) are taken kWBatch at a time; their weights, phases r and
// e^{2 pi i delta j / L} are formed once per block in shared memory, and each bin adds
// w e^{2 pi i k r / S} e^{2 pi i delta j / L} in FP64. Bound by the FP64 pipe (about two
// FMAs a clock and SM): 0.3 ms at 65536 samples, 144 bins and two trajectories, against
// some 0.1 s on the host's cores.
constexpr int kWBatch = 32;

struct FoldTraj {
    const int *csr_ptr;
    const CsrEntry *csr;
    const int2 *tnf;           // (cell n, -) per sample
    const double *drive;       // [S] A sin(2 pi r / S + phi0)
    const double *vel;         // [n_par][S]
    const double2 *unit_s;     // [S] e^{2 pi i m / S}
    const float2 *dgam;
    double slope;              // (N - 1) / (L - 1)
};

__global__ void __launch_bounds__(256) k_fold_w(FoldTraj T, double *__restrict__ W, Dims d) {
    extern __shared__ double fw_sm[];  // [kWBatch][W] (cos, sin) pairs, then [kWBatch] weights
    double2 *ph = reinterpret_cast<double2 *>(fw_sm);
    double *wt = fw_sm + 2 * kWBatch * d.W;
    int *rr = reinterpret_cast<int *>(wt + kWBatch);
    const int e = blockIdx.x, par = blockIdx.y;
    const int *ptr = T.csr_ptr + (size_t)par * (d.Ne + 1);
    const CsrEntry *ent = T.csr + (size_t)par * 2 * d.L;
    const int k0 = ptr[e], k1 = ptr[e + 1];
    for (int o0 = 0; o0 < d.nb; o0 += blockDim.x) {  // uniform trip count
        const int o = o0 + threadIdx.x;
        const int kh = d.kmin + o / d.W, di = o % d.W;
        double ar = 0.0, ai = 0.0;
        for (int kb = k0; kb < k1; kb += kWBatch) {
            const int n = min(kWBatch, k1 - kb);
            __syncthreads();  // the previous batch has been used
            for (int t = threadIdx.x; t < n * d.W; t += blockDim.x) {
                const int q = t / d.W, dd = t - q * d.W;
                const int j = ent[kb + q].j;
                long long num = (long long)(dd - d.hw) * j % d.L;
                if (num < 0) num += d.L;
                double s, c;
                sincospi(2.0 * (double)num / (double)d.L, &s, &c);
                ph[t] = make_double2(c, s);
                if (dd == 0) {
                    const int r = j % d.S, cell = T.tnf[(size_t)par * d.L + j].x;
                    const double slow = par ? (double)(d.N - 1) - T.slope * j : T.slope * j;
                    const double f = (double)d.Q * (slow + T.drive[r]) + (double)d.D - (double)cell;
                    wt[q] = T.vel[(size_t)par * d.S + r] * (cell == e ? 1.0 - f : f);
                    rr[q] = r;
                }
            }
            __syncthreads();
            if (o < d.nb)
                for (int q = 0; q < n; ++q) {
                    const double2 u = T.unit_s[(int)((long long)kh * rr[q] % d.S)];
                    const double2 p = ph[q * d.W + di];
                    ar = fma(wt[q], u.x * p.x - u.y * p.y, ar);
                    ai = fma(wt[q], u.x * p.y + u.y * p.x, ai);
                }
        }
        if (o < d.nb) {
            const double isl = 1.0 / sqrt((double)d.L);
            const float2 g = T.dgam[o];
            double *out = W + ((size_t)par * 2 * d.nb + 2 * o) * d.Ne + e;
            out[0] = isl * ((double)g.x * ar - (double)g.y * ai);
            out[d.Ne] = isl * ((double)g.x * ai + (double)g.y * ar);
        }
    }
}

// out[par][z][o][i] = sum_e W[par][o][e] g[z][e - D - Q i - kmin]: a warp takes one row o and 32
// columns i, a block two rows of one z and trajectory; e runs in tiles of 256 staged in shared
// memory with the taps they meet, which lie there by residue modulo Q, so that the lanes of a
// warp (taps Q apart) read neighbouring words. Bound by the FP64 pipe, two FMAs a clock and SM:
// small blocks spread even one small fold over the GPU. With eight rows and 128 columns a block a
// fold at 32^2 x 16 ran on 12 SMs and took 160 us.
constexpr int kWdRows = 2, kWdCols = 32, kWdTile = 256;

__global__ void __launch_bounds__(32 * kWdRows) k_fold_taps(const double *__restrict__ W,
                                                            const double *__restrict__ g, double *__restrict__ out,
                                                            int R, int Ne, int N, int Nz, int D, int Q, int kmin,
                                                            int Lk) {
    __shared__ double sw[kWdRows][kWdTile];
    __shared__ double sg[kWdTile + 32 * kWdCols];  // [Q][kWdTile / Q + kWdCols] taps, Q <= 32
    const int ncb = (N + kWdCols - 1) / kWdCols;
    const int o0 = (blockIdx.x / ncb) * kWdRows, i0 = (blockIdx.x % ncb) * kWdCols;
    const int d = blockIdx.y, par = blockIdx.z;
    const int lane = threadIdx.x & 31, r = threadIdx.x >> 5, i = i0 + lane;
    const double *Wp = W + (size_t)par * R * Ne;
    const double *gd = g + (size_t)d * Lk;
    const int per = kWdTile / Q + kWdCols, span = kWdTile + Q * (kWdCols - 1);
    double acc = 0.0;
    for (int e0 = 0; e0 < Ne; e0 += kWdTile) {
        __syncthreads();
        for (int t = threadIdx.x; t < kWdRows * kWdTile; t += blockDim.x) {
            const int rr = t / kWdTile, e = e0 + t % kWdTile;
            sw[rr][t % kWdTile] = (o0 + rr < R && e < Ne) ? Wp[(size_t)(o0 + rr) * Ne + e] : 0.0;
        }
        // k = e - D - Q i runs from kb (e = e0, i = i0 + kWdCols - 1) upwards
        const int kb = e0 - D - Q * (i0 + kWdCols - 1) - kmin;
        for (int t = threadIdx.x; t < span; t += blockDim.x) {
            const int k = kb + t;
            sg[(t % Q) * per + t / Q] = (k >= 0 && k < Lk) ? gd[k] : 0.0;
        }
        __syncthreads();
        const double *gl = sg + kWdCols - 1 - lane;
        for (int b = 0; b < kWdTile / Q; ++b)
            for (int q = 0; q < Q; ++q) acc = fma(sw[r][b * Q + q], gl[q * per + b], acc);
    }
    if (i < N && o0 + r < R) out[(((size_t)par * Nz + d) * R + o0 + r) * N + i] = acc;
}

// FP32 operands of the staged path from W H [n_par][ns][2 n_b][N], z = blockIdx.z of ns:
// f_z[par][i][o] (columns past 2 n_b zero) and, of slot 0, a[par][o][i] (columns past N zero)
__global__ void __launch_bounds__(256) k_fold_operands(const double *__restrict__ WH, float *__restrict__ f0,
                                                       float *__restrict__ f1, float *__restrict__ a, int R, int N,
                                                       int ldf, int lda) {
    const int par = blockIdx.y;
    const double *src = WH + ((size_t)par * gridDim.z + blockIdx.z) * R * N;
    float *f = blockIdx.z ? f1 : f0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < N * ldf; t += gridDim.x * blockDim.x) {
        const int i = t / ldf, o = t - i * ldf;
        f[(size_t)par * N * ldf + t] = o < R ? (float)src[(size_t)o * N + i] : 0.f;
    }
    if (!a || blockIdx.z) return;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < R * lda; t += gridDim.x * blockDim.x) {
        const int o = t / lda, i = t - o * lda;
        a[(size_t)par * R * lda + t] = i < N ? (float)src[(size_t)o * N + i] : 0.f;
    }
}

FoldState *state(mpi_ffl_handle *h) {
    if (!h->fold_state) h->fold_state = new FoldState();
    return fs(h);
}

// Taps of both slots at offsets (kmin + k) / Q on the device, for the handle's width
int taps_ready(mpi_ffl_handle *h) {
    FoldState *s = fs(h);
    if (s->taps_fwhm == h->fwhm) return MPI_FFL_OK;
    const Dims &d = h->d;
    const int n = fold_taps(d);
    if (!falloc(&s->taps, 2 * (size_t)n)) return MPI_FFL_ERR_OOM;
    std::vector<double> g(2 * (size_t)n);
    for (int k = 0; k < n; ++k) {
        g[k] = h->taps.h[std::abs(k + fold_kmin(d))];
        g[n + k] = h->taps.dh[std::abs(k + fold_kmin(d))];
    }
    s->taps_fwhm = -1.0;
    if (!fupload(s->taps, g)) return MPI_FFL_ERR_CUDA;
    s->taps_fwhm = h->fwhm;
    return MPI_FFL_OK;
}

// W H of slots [first, first + n) into s->WH
int fold_slots(mpi_ffl_handle *h, int first, int n, cudaStream_t st) {
    const Dims &d = h->d;
    int rc = fold_w(h);
    if (rc == MPI_FFL_OK) rc = taps_ready(h);
    if (rc != MPI_FFL_OK) return rc;
    FoldState *s = fs(h);
    if (!falloc(&s->WH, (size_t)d.n_par * 2 * 2 * d.nb * d.N)) return MPI_FFL_ERR_OOM;
    launch_fold_taps(s->W, s->taps + (size_t)first * fold_taps(d), s->WH, d, d.n_par, n, st);
    return MPI_FFL_OK;
}

bool capturing(cudaStream_t st) {
    cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &c) != cudaSuccess) cudaGetLastError();  // the legacy stream, which cannot be
    return c == cudaStreamCaptureStatusActive;
}

// The operands of slots [first, first + n), whose buffers are there. Under capture the fold
// becomes part of the graph, whose replays then fold too, and the slot does not count as ready.
int refold(mpi_ffl_handle *h, int first, int n, cudaStream_t st) {
    const Dims &d = h->d;
    const int rc = fold_slots(h, first, n, st);
    if (rc != MPI_FFL_OK) return rc;
    FoldState *s = fs(h);
    const int R = 2 * d.nb, work = std::max(d.N * s->ldf, R * s->lda);
    k_fold_operands<<<dim3(std::min(608, (work + 255) / 256), d.n_par, n), 256, 0, st>>>(
        s->WH, s->f[first], s->f[1], first == 0 ? s->a : nullptr, R, d.N, s->ldf, s->lda);
    if (capturing(st)) return MPI_FFL_OK;
    // another stream may use the operands next
    if (cudaStreamSynchronize(st) != cudaSuccess) return MPI_FFL_ERR_CUDA;
    for (int k = first; k < first + n; ++k) s->ready[k] = s->used[k] = true;
    return MPI_FFL_OK;
}

}  // namespace

namespace {

// W of a small scan (at most kHostW values) on the host, sample by sample: 3 to 6 ms on the
// thread that prepares a request, beside the running batch, without the temporary device
// memory of the device build, whose release waits for the batch. The device build takes 0.6
// ms at these sizes. No measurement favours the host here: with the device build a tiny request
// is done 9 ms after its arrival, and requests 10 ms apart no longer meet in the server, which
// tests/test_gpu_serving.py holds it to (it failed in three of six runs). The line lies between
// that test's largest scan (40082 values) and the next size in use (48080).
constexpr size_t kHostW = 40960;

std::vector<double> w_host(const mpi_ffl_handle *h) {
    const Dims &d = h->d;
    const double kPi = 3.14159265358979323846;
    const size_t R = (size_t)2 * d.nb;
    const double isl = 1.0 / std::sqrt((double)d.L);
    std::vector<double> W(d.n_par * R * d.Ne, 0.0), cs(d.S), sn(d.S);
    for (int m = 0; m < d.S; ++m) {
        cs[m] = std::cos(2.0 * kPi * m / d.S);
        sn[m] = std::sin(2.0 * kPi * m / d.S);
    }
    for (int par = 0; par < d.n_par; ++par)
        for (int j = 0; j < d.L; ++j) {
            int n;
            double f, v;
            traj_point_host(h, par, j, n, f, v);
            for (int di = 0; di < d.W; ++di) {
                const int64_t dl = di - d.hw;
                const double ad = 2.0 * kPi * (double)(((dl * j) % d.L + d.L) % d.L) / d.L;
                const double cd = std::cos(ad), sd = std::sin(ad);
                for (int k = 0; k < d.K; ++k) {
                    // e^{2 pi i (kP + delta) j / L} = e^{2 pi i k r / S} e^{2 pi i delta j / L}
                    const int m = (int)((int64_t)(d.kmin + k) * (j % d.S) % d.S);
                    const double ck = cs[m], sk = sn[m];
                    const double er = ck * cd - sk * sd, ei = ck * sd + sk * cd;
                    const int o = k * d.W + di;
                    const double gr = h->dgamma[2 * o], gi = h->dgamma[2 * o + 1];
                    const double wr = (gr * er - gi * ei) * isl, wi = (gr * ei + gi * er) * isl;
                    double *row = W.data() + (par * R + 2 * o) * d.Ne + n;
                    row[0] += (1.0 - f) * v * wr;
                    row[d.Ne] += (1.0 - f) * v * wi;
                    row[1] += f * v * wr;
                    row[d.Ne + 1] += f * v * wi;
                }
            }
        }
    return W;
}

}  // namespace

int fold_w(mpi_ffl_handle *h) {
    FoldState *s = state(h);
    if (s->W) return MPI_FFL_OK;
    const Dims &d = h->d;
    const double kPi = 3.14159265358979323846;
    if ((size_t)2 * d.nb * d.Ne <= kHostW) {
        const std::vector<double> W = w_host(h);
        if (!falloc(&s->W, W.size())) return MPI_FFL_ERR_OOM;
        if (fupload(s->W, W)) return MPI_FFL_OK;
        dev_free(s->W);  // not filled: the next call builds it
        s->W = nullptr;
        return MPI_FFL_ERR_CUDA;
    }
    double *drive = nullptr, *vel = nullptr, *W = nullptr;
    double2 *unit_s = nullptr;
    const bool ok = falloc(&drive, d.S) && falloc(&vel, (size_t)d.n_par * d.S) && falloc(&unit_s, d.S) &&
                    falloc(&W, (size_t)d.n_par * 2 * d.nb * d.Ne);
    int rc = ok ? MPI_FFL_OK : MPI_FFL_ERR_OOM;
    if (ok) {
        std::vector<double> hd(d.S), hv((size_t)d.n_par * d.S);
        std::vector<double2> hu(d.S);
        const double slope = (double)(d.N - 1) / (double)(d.L - 1);
        for (int r = 0; r < d.S; ++r) {
            const double ph = 2.0 * kPi * r / d.S + h->phase;
            hd[r] = h->amp * std::sin(ph);
            for (int par = 0; par < d.n_par; ++par)
                hv[(size_t)par * d.S + r] = (par ? -slope : slope) + h->amp * (2.0 * kPi / d.S) * std::cos(ph);
            hu[r] = make_double2(std::cos(2.0 * kPi * r / d.S), std::sin(2.0 * kPi * r / d.S));
        }
        cudaMemcpy(drive, hd.data(), hd.size() * sizeof(double), cudaMemcpyHostToDevice);
        cudaMemcpy(vel, hv.data(), hv.size() * sizeof(double), cudaMemcpyHostToDevice);
        cudaMemcpy(unit_s, hu.data(), hu.size() * sizeof(double2), cudaMemcpyHostToDevice);
        const FoldTraj T{h->t_csr_ptr, h->t_csr, h->t_tnf, drive, vel, unit_s, h->t_dgam, slope};
        const size_t smem = sizeof(double) * (2 * kWBatch * d.W + kWBatch) + sizeof(int) * kWBatch;
        const int threads = std::min(256, (d.nb + 31) / 32 * 32);
        k_fold_w<<<dim3(d.Ne, d.n_par), threads, smem>>>(T, W, d);
        if (cudaStreamSynchronize(nullptr) != cudaSuccess) rc = MPI_FFL_ERR_CUDA;
    }
    for (void *p : {(void *)drive, (void *)vel, (void *)unit_s})
        if (p) dev_free(p);
    if (rc == MPI_FFL_OK) s->W = W;
    else if (W) dev_free(W);
    return rc;
}

const double *fold_w_dev(const mpi_ffl_handle *h) { return fs(h) ? fs(h)->W : nullptr; }

void launch_fold_taps(const double *W, const double *g, double *out, const Dims &d, int n_par, int nz,
                      cudaStream_t st) {
    const int R = 2 * d.nb, ncb = (d.N + kWdCols - 1) / kWdCols;
    k_fold_taps<<<dim3(((R + kWdRows - 1) / kWdRows) * ncb, nz, n_par), 32 * kWdRows, 0, st>>>(
        W, g, out, R, d.Ne, d.N, nz, d.D, d.Q, fold_kmin(d), fold_taps(d));
}

const double *fold_wh(mpi_ffl_handle *h, cudaStream_t st) {
    return fold_slots(h, 0, 1, st) == MPI_FFL_OK ? fs(h)->WH : nullptr;
}

// The folded stage costs 2 n_b N FMAs a line, the stage kernels N N_e (H), about
// L (2 w + 3) (resampling and band DFT) and the signal's way through HBM: the stages are
// cheaper only for short lines with wide bands. W is kept in FP64 (at most 512 MB). With
// the stages an FP32 pair took 1617 us at 256^2 x 128 and 36 angles, 299 us at 128^2 x 64
// and 24; folded 276 and 70 us, with smaller errors against 64 bits (one rounded matrix in
// the place of rounded taps, weights and twiddles). A band of 2 n_b = 180 and lines of 256
// samples on 20 bins (N_e = 109) is on the other side of the line.
bool fold_fits(const Dims &d) {
    const double folded = 2.0 * d.nb * d.N, staged = (double)d.N * d.Ne + (double)d.L * (d.W + 2);
    return folded <= staged && (double)d.n_par * 2 * d.nb * d.Ne * sizeof(double) <= 512e6;
}

namespace {

// the staged path's lines and buffers, of both slots: the first gradient may be captured after a
// forward outside
int staged_buffers(mpi_ffl_handle *h) {
    const Dims &d = h->d;
    FoldState *s = fs(h);
    if (!s->rows) {
        std::vector<int> rows;
        for (int par = 0; par < d.n_par; ++par) {
            for (int m = 0; m < d.M; ++m)
                for (int z = par; z < d.Nz; z += d.n_par) rows.push_back(m * d.Nz + z);
            s->nrows[par] = (int)rows.size() - (par ? s->nrows[0] : 0);
        }
        if (!falloc(&s->rows, rows.size())) return MPI_FFL_ERR_OOM;
        if (!fupload(s->rows, rows)) {
            dev_free(s->rows);
            s->rows = nullptr;
            return MPI_FFL_ERR_CUDA;
        }
    }
    const int R = 2 * d.nb;
    s->ldf = (R + 3) / 4 * 4;
    s->lda = (d.N + 3) / 4 * 4;
    const size_t f_len = (size_t)d.n_par * d.N * s->ldf;
    return falloc(&s->f[0], f_len) && falloc(&s->f[1], f_len) && falloc(&s->a, (size_t)d.n_par * R * s->lda)
               ? MPI_FFL_OK
               : MPI_FFL_ERR_OOM;
}

}  // namespace

int fold_ready(mpi_ffl_handle *h, int slot, cudaStream_t st) {
    FoldState *s = state(h);
    if (s->ready[slot]) return MPI_FFL_OK;
    int rc = staged_buffers(h);
    if (rc == MPI_FFL_OK) rc = refold(h, slot, 1, st);
    if (rc != MPI_FFL_OK) fold_trim(h);
    return rc;
}

// Nothing of a failed build is kept: without operands of the staged path or of the collapsed
// operator in use the next call builds all of it again.
void fold_trim(mpi_ffl_handle *h) {
    const FoldState *s = fs(h);
    if (s && !s->used[0] && !s->used[1] && !col_supported(h)) fold_release(h);
}

void fold_forward(mpi_ffl_handle *h, int slot, const float *proj, const float *gain, float *data, cudaStream_t st) {
    const Dims &d = h->d;
    const FoldState *s = fs(h);
    SgemmArgs g[2];
    for (int par = 0; par < d.n_par; ++par) {
        const int *rows = s->rows + (par ? s->nrows[0] : 0);
        g[par] = SgemmArgs{proj, d.N,      rows, s->nrows[par], d.N,  s->f[slot] + (size_t)par * d.N * s->ldf,
                           s->ldf, data,   2 * d.nb, rows,      2 * d.nb, gain, d.Nz, nullptr, nullptr};
    }
    launch_sgemm(g, d.n_par, st);
}

void fold_adjoint(mpi_ffl_handle *h, const float *data, const float *gain, float *proj, cudaStream_t st) {
    const Dims &d = h->d;
    const FoldState *s = fs(h);
    const int R = 2 * d.nb;
    SgemmArgs g[2];
    for (int par = 0; par < d.n_par; ++par) {
        const int *rows = s->rows + (par ? s->nrows[0] : 0);
        g[par] = SgemmArgs{data, R,    rows, s->nrows[par], R,   s->a + (size_t)par * R * s->lda,
                           s->lda, proj, d.N, rows,          d.N, gain, d.Nz, nullptr, nullptr};
        // The rows of W H fall off with the harmonic: from the last to the first, a sum has its size
        // only at the end. Error of the adjoint against 64 bits at 256^2 x 128 and 36 angles 1.7e-7
        // (3.1e-7 from the first on, 1.9e-7 through the separate stages), at 64^2 x 32 1.2e-7
        // (1.9e-7, 1.3e-7).
        g[par].back = true;
    }
    launch_sgemm(g, d.n_par, st);
}

void fold_psf_changed(mpi_ffl_handle *h) {
    if (FoldState *s = fs(h)) s->ready[0] = s->ready[1] = false;
}

void fold_refresh(mpi_ffl_handle *h) {
    const FoldState *s = fs(h);
    if (!s) return;
    const bool need[2] = {s->used[0] && !s->ready[0], s->used[1] && !s->ready[1]};
    if (!need[0] && !need[1]) return;
    try {
        refold(h, need[0] ? 0 : 1, need[0] && need[1] ? 2 : 1, nullptr);
    } catch (...) {  // a host allocation
    }
}

BufferList fold_buffers(const mpi_ffl_handle *h) {
    const FoldState *s = fs(h);
    if (!s) return {};
    return {s->W, s->taps, s->WH, s->f[0], s->f[1], s->a, s->rows};
}

void fold_release(mpi_ffl_handle *h) {
    FoldState *s = fs(h);
    if (!s) return;
    for (void *p : fold_buffers(h)) dev_free(p);
    delete s;
    h->fold_state = nullptr;
}

}  // namespace mpiffl
