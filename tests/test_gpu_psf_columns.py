"""H and its transpose where lines go one at a time and not in pairs: columns along z so long that
two of them do not fit a block's shared memory beside the taps, and numbers of lines that pairs
would spread unevenly."""

import numpy as np
import pytest

from _helpers import OP_TOL, ensure_library, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Setup, psf, zdrive  # noqa: E402
from oracle.data import to_interleaved  # noqa: E402

GEOM = dict(nx=8, n_angles=2, A=4.0, phi0=0.2, zigzag=1, fwhm=3.0, k_min=1, half_width=1)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_library()


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


# Q = 32: pairs of columns up to 420 slices; 512 and 560 slices go alone, an odd number of columns
@pytest.mark.parametrize("nx,nz", [(8, 420), (8, 512), (7, 560)])
def test_long_columns_and_their_transpose(nx, nz):
    from paper_2511_06627_gb300 import FFLOperator

    geom = dict(GEOM, nx=nx, nz=nz, S=16, P=10, Q=32, k_max=4)
    st, op = Setup(**geom), FFLOperator(**geom)
    rng = np.random.default_rng(51)
    proj = rng.standard_normal((st.n_angles, nz, nx)).astype(np.float32)
    cz = rng.standard_normal((st.n_angles, nx, zdrive.n_fine_z(st))).astype(np.float32)
    assert rel_l2(op.apply_stage_zdrive(1, _t(proj)).cpu().numpy(), zdrive.psf_fwd_z(proj, st)) < OP_TOL
    assert rel_l2(op.apply_stage_zdrive(1, _t(cz), transpose=True).cpu().numpy(), zdrive.psf_adj_z(cz, st)) < OP_TOL
    m = np.array([1])
    y = np.zeros(st.data_shape, dtype=np.complex64)
    y[m] = rng.standard_normal(y[m].shape) + 1j * rng.standard_normal(y[m].shape)
    x = rng.standard_normal((nz, nx, nx)).astype(np.float32)
    got = op.forward_zdrive(_t(x)).cpu().numpy()[m]  # few periods a column: the sampled kernels
    assert rel_l2(got, to_interleaved(zdrive.forward_stages_z(x, st, angles=m)["data"])) < OP_TOL
    got = op.adjoint_zdrive(_t(to_interleaved(y))).cpu().numpy()
    assert rel_l2(got, zdrive.adjoint_stages_z(y[m], st, angles=m)["vol"]) < OP_TOL
    op.sync_check()
    op.close()


def test_a_column_beyond_the_shared_memory_is_refused():
    """600 slices at Q = 32: one column and the taps need 236 KB."""
    from paper_2511_06627_gb300 import FFLOperator, MpiFflError

    geom = dict(GEOM, nx=7, nz=600, S=16, P=10, Q=32, k_max=4)
    op = FFLOperator(**geom)
    with pytest.raises(MpiFflError):
        op.apply_stage_zdrive(1, torch.zeros(op.n_angles, 7, op.fine_len_z, device="cuda"), transpose=True)
    op.close()


def test_a_column_of_ten_thousand_slices():
    """Q = 2: H alone, at some of its fine points."""
    from paper_2511_06627_gb300 import FFLOperator

    geom = dict(GEOM, nx=2, n_angles=1, nz=10001, S=4, P=8, Q=2, k_max=1, half_width=0)
    st, op = Setup(**geom), FFLOperator(**geom)
    rng = np.random.default_rng(52)
    proj = rng.standard_normal((1, st.nz, 2)).astype(np.float32)
    got = op.apply_stage_zdrive(1, _t(proj)).cpu().numpy()[0]  # [u][e]
    e = np.unique(np.concatenate([rng.integers(0, zdrive.n_fine_z(st), 300), [0, zdrive.n_fine_z(st) - 1]]))
    h = psf.h((e[:, None] - st.D) / st.Q - np.arange(st.nz)[None, :], st.fwhm)
    assert rel_l2(got[:, e], (h @ proj[0].astype(np.float64)).T) < OP_TOL
    op.close()


# lines in pairs and one at a time, by the blocks on the fullest SM: H in pairs and H^T not, the
# reverse, both singly, both in pairs; lines that are no multiple of a block's; other numbers of lanes
@pytest.mark.parametrize("nx,nz,M,Q", [(40, 64, 24, 8), (33, 41, 13, 8), (64, 23, 9, 8), (35, 96, 21, 8),
                                       (30, 61, 25, 4), (21, 51, 12, 16), (19, 70, 30, 2)])
def test_lines_in_pairs_and_singly(nx, nz, M, Q):
    from paper_2511_06627_gb300 import FFLOperator

    geom = dict(GEOM, nx=nx, nz=nz, n_angles=M, S=16, P=20, Q=Q, k_max=4)
    st, op = Setup(**geom), FFLOperator(**geom)
    h = psf.h((np.arange(st.n_fine)[:, None] - st.D) / st.Q - np.arange(nx)[None, :], st.fwhm)
    rng = np.random.default_rng(53)
    p = rng.standard_normal((M, nz, nx)).astype(np.float32)
    f = rng.standard_normal((M, nz, st.n_fine)).astype(np.float32)
    assert rel_l2(op.apply_stage(1, _t(p)).cpu().numpy(), p @ h.T) < OP_TOL
    assert rel_l2(op.apply_stage(1, _t(f), transpose=True).cpu().numpy(), f @ h) < OP_TOL
    op.close()
