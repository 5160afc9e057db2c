// The line operator of one trajectory folded to a matrix in FP64 on the device, and the
// FP32 matrix products that apply it (fold.cu).
#pragma once

#include "internal.h"

namespace mpiffl {

// FP64 matrices, one per trajectory: W = S D_Gamma F V E ([2 n_b][N_e], rows alternating
// Re and Im of the kept bins) and taps applied to it, W T ([2 n_b][N]) with
// T[e][i] = taps[e - D - Q i - kmin].
int fold_w(mpi_ffl_handle *h);                  // builds W on first use; MPI_FFL_OK or an error
const double *fold_w_dev(const mpi_ffl_handle *h);  // [n_par][2 n_b][N_e], after fold_w
// first index k = e - D - Q i of the taps and their count
inline int fold_kmin(const Dims &d) { return -d.D - d.Q * (d.N - 1); }
inline int fold_taps(const Dims &d) { return d.Ne + d.Q * (d.N - 1); }
// out[par][z][o][i] = sum_e W[par][o][e] g[z][e - D - Q i - kmin], z < nz, on the stream
void launch_fold_taps(const double *W, const double *g, double *out, const Dims &d, int n_par, int nz,
                      cudaStream_t st);
// W H in FP64 ([n_par][2 n_b][N]) for the handle's PSF, valid until the next call or refold;
// NULL when an allocation failed
const double *fold_wh(mpi_ffl_handle *h, cudaStream_t st);

// Staged path: W H in FP32, applied to the projections (forward) or to the data (adjoint).
bool fold_fits(const Dims &d);                  // the rule by sizes
int fold_ready(mpi_ffl_handle *h, int slot, cudaStream_t st);  // operands built on first use
void fold_forward(mpi_ffl_handle *h, int slot, const float *proj, const float *gain, float *data, cudaStream_t st);
void fold_adjoint(mpi_ffl_handle *h, const float *data, const float *gain, float *proj, cudaStream_t st);
void fold_psf_changed(mpi_ffl_handle *h);       // marks the operands as stale
// Refolds the stale operands of the slots that calls have used. Those it could not refold are left to their next use, which
// tries again and reports.
void fold_refresh(mpi_ffl_handle *h);
void fold_trim(mpi_ffl_handle *h);              // after a failed build: releases what nothing uses
BufferList fold_buffers(const mpi_ffl_handle *h);  // its device allocations
void fold_release(mpi_ffl_handle *h);

// C[crow[i]][ccol[n]] = scale[arow[i] / rdiv] sum_k A[arow[i]][acol[k]] B[k][n] in FP32
// (arow, crow, acol and ccol may be NULL: row i, column k or n; scale NULL: 1). B is K x
// ldb, ldb a multiple of 4, on 16 bytes; its rows hold bcols values that may be read (a
// multiple of 4; 0: ldb). nbatch: that many such products, their operands sA, sB (a
// multiple of 4) and sC values apart. half > 0: two products E and O of half values of k
// each, O's in columns ahalf (a multiple of 4) and rows bhalf further on; E + O goes to
// column n, E - O to column c1 + n, or c1 - n when mirror is set (no acol and ccol, one batch).
// back: k is summed from the last stage of 16 to the first (not with half). fine: in short runs.
struct SgemmArgs {
    const float *A = nullptr;
    int64_t lda = 0;
    const int *arow = nullptr;
    int M = 0, K = 0;
    const float *B = nullptr;
    int ldb = 0;
    float *C = nullptr;
    int64_t ldc = 0;
    const int *crow = nullptr;
    int N = 0;
    const float *scale = nullptr;
    int rdiv = 1;
    const int *acol = nullptr, *ccol = nullptr;
    int nbatch = 1, bcols = 0;
    int64_t sA = 0, sB = 0, sC = 0;
    int half = 0, ahalf = 0, bhalf = 0, c1 = 0;
    bool mirror = false;
    bool back = false, fine = false;
};
constexpr int kSgemmMax = 9;  // problems of one launch
void launch_sgemm(const SgemmArgs *g, int n, cudaStream_t st);
int sgemm_tiles(const SgemmArgs &g);  // its blocks with the largest tiles

// The z-drive scan with the raster and the PSF along z folded to tables (k_zfold.cu).
bool zfold_fits(const Dims &d);                      // the rule by sizes
int zfold_ready(mpi_ffl_handle *h);                  // tables and workspace, on first use
void zfold_forward(mpi_ffl_handle *h, const float *proj, float *data, cudaStream_t st);
void zfold_adjoint(mpi_ffl_handle *h, const float *data, float *proj, cudaStream_t st);
// Rebuilds the table of the width, or leaves it to its next use, which tries again and reports.
void zfold_psf_changed(mpi_ffl_handle *h);
BufferList zfold_buffers(const mpi_ffl_handle *h);
void zfold_release(mpi_ffl_handle *h);

}  // namespace mpiffl
