"""Line stages at the sizes where their kernels' layouts change, against the FP64 oracle."""

import numpy as np
import pytest

from _helpers import OP_TOL, ensure_library, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Setup, operator  # noqa: E402
from oracle.data import to_interleaved  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_library()


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _n(t):
    torch.cuda.synchronize()
    return t.detach().cpu().numpy().astype(np.float64)


def _make(**kw):
    from paper_2511_06627_gb300 import FFLOperator

    geom = dict(dict(nx=20, nz=5, n_angles=3, S=10, P=15, A=4.0, phi0=0.2, zigzag=1, Q=4, fwhm=2.5, k_min=1, k_max=3,
                     half_width=1), **kw)
    return Setup(**geom), FFLOperator(**geom)


@pytest.mark.parametrize("S,P", [(10, 15), (14, 9), (132, 7), (10, 16)])
def test_band_dft_with_an_odd_number_of_periods(S, P):
    """P (2w + 1) floats of twiddles are odd when P is: the complex values after them in
    shared memory still start on 8 bytes (periods of S not a multiple of 4, or above 128)."""
    st, op = _make(S=S, P=P)
    rng = np.random.default_rng(5)
    sig = rng.standard_normal((st.n_angles, st.nz, st.L)).astype(np.float32)
    assert rel_l2(_n(op.apply_stage(3, _t(sig))), to_interleaved(operator.compress_fwd(sig, st))) < OP_TOL
    y = (rng.standard_normal(st.data_shape) + 1j * rng.standard_normal(st.data_shape)).astype(np.complex64)
    got = _n(op.apply_stage(3, _t(to_interleaved(y)), transpose=True))
    assert rel_l2(got, operator.compress_adj(y, st)) < OP_TOL


# the staged path's folded line stage: both tile sizes of its matrix product with ragged
# edges, one trajectory and two, and a short line with a wide band, which keeps the stages
STAGED = {
    "ragged": dict(nx=33, nz=7, n_angles=5, S=12, P=40, k_max=4, half_width=2),
    "one trajectory": dict(nx=38, nz=9, n_angles=4, zigzag=0, S=16, P=33, k_max=6, half_width=0),
    "large tiles": dict(nx=50, nz=129, n_angles=26, S=16, P=50, k_max=6, half_width=4),
    "stages": dict(nx=20, nz=6, n_angles=3, S=64, P=4, k_max=30, half_width=1),
}


@pytest.mark.parametrize("name", list(STAGED))
def test_staged_path_against_the_oracle(name):
    st, op = _make(**STAGED[name])
    rng = np.random.default_rng(6)
    gains = (1 + 0.1 * rng.standard_normal(st.n_angles)).astype(np.float32)
    op.set_gain(gains)
    st.gains = gains.astype(np.float64)
    m = np.array([st.n_angles - 1])  # one angle is enough to place every line
    x = rng.standard_normal((st.nz, st.nx, st.nx)).astype(np.float32)
    y = np.zeros(st.data_shape, dtype=np.complex64)
    y[m] = rng.standard_normal(y[m].shape) + 1j * rng.standard_normal(y[m].shape)
    for fwhm in (2.5, 3.25):  # the second width refolds the operands
        op.set_fwhm(fwhm)
        st.fwhm = fwhm
        ref = operator.forward_stages(x, st, angles=m)
        assert rel_l2(_n(op.forward(_t(x)))[m], to_interleaved(ref["data"])) < OP_TOL
        assert rel_l2(_n(op.adjoint(_t(to_interleaved(y)))), operator.adjoint_stages(y[m], st, angles=m)["vol"]) < OP_TOL
        dfine = ref["proj"] @ operator.psf.dh_dfwhm((np.arange(st.n_fine)[:, None] - st.D) / st.Q
                                                     - np.arange(st.nx)[None, :], fwhm).T
        db = operator.compress_fwd(operator.resample_fwd(dfine, st, m), st)
        gb = np.zeros(st.data_shape, dtype=np.complex64)
        gb[m] = db  # the width gradient's inner product without cancellation
        gg, gw = op.param_grad(_t(x), _t(to_interleaved(gb)))
        assert abs(float(gw) / np.vdot(gb[m], db).real - 1) < 2 * OP_TOL
        bare = np.vdot(gb[m], ref["data"] / gains[m[0]]).real
        assert abs(float(gg[m[0]]) - bare) < OP_TOL * np.linalg.norm(gb) * np.linalg.norm(ref["data"])
    op.close()


# the z-drive scan: folded tables with odd phases, harmonics and slices, one trajectory and
# two, both convolution widths, more phases than a block has threads; and a raster with few
# periods a column, which keeps the sample-by-sample kernels
ZDRIVE = {
    "odd": dict(nx=21, nz=9, n_angles=3, S=15, P=30, k_max=5, half_width=1),
    "one trajectory": dict(nx=18, nz=11, n_angles=2, zigzag=0, S=24, P=20, k_max=4, half_width=2),
    "sixteen lines": dict(nx=24, nz=67, n_angles=60, S=16, P=40, k_max=3, half_width=1),
    "many phases": dict(nx=16, nz=5, n_angles=2, S=140, P=20, k_max=7, half_width=0),
    "sampled": dict(nx=40, nz=8, n_angles=3, S=32, P=6, k_max=5, half_width=1),
    # the products by K in halves of the columns (scans that fill the GPU): odd and not a
    # multiple of four, odd slices, no harmonic offsets; and the large tiles of both products
    "odd columns in halves": dict(nx=23, nz=95, n_angles=64, S=64, P=30, k_max=5, half_width=1),
    "66 columns": dict(nx=66, nz=96, n_angles=64, S=60, P=70, k_max=6, half_width=0),
    "large halves": dict(nx=19, nz=112, n_angles=60, S=128, P=20, k_max=5, half_width=3),
}


@pytest.mark.parametrize("name", list(ZDRIVE))
def test_zdrive_against_the_oracle(name):
    from oracle import zdrive

    st, op = _make(**ZDRIVE[name])
    rng = np.random.default_rng(7)
    gains = (1 + 0.1 * rng.standard_normal(st.n_angles)).astype(np.float32)
    op.set_gain(gains)
    st.gains = gains.astype(np.float64)
    m = np.array([st.n_angles - 1])
    x = rng.standard_normal((st.nz, st.nx, st.nx)).astype(np.float32)
    y = np.zeros(st.data_shape, dtype=np.complex64)
    y[m] = rng.standard_normal(y[m].shape) + 1j * rng.standard_normal(y[m].shape)
    for fwhm in (2.5, 3.25):
        op.set_fwhm(fwhm)
        st.fwhm = fwhm
        ref = zdrive.forward_stages_z(x, st, angles=m)["data"]
        assert rel_l2(_n(op.forward_zdrive(_t(x)))[m], to_interleaved(ref)) < OP_TOL
        assert rel_l2(_n(op.adjoint_zdrive(_t(to_interleaved(y)))), zdrive.adjoint_stages_z(y[m], st, angles=m)["vol"]) < OP_TOL
    op.close()


@pytest.mark.parametrize("nx,nz,off", [(21, 9, 0), (102, 8, 0), (259, 3, 0), (64, 9, 1), (33, 5, 3)])
def test_interleaved_projector_on_ragged_detectors(nx, nz, off):
    """Detectors that are not a multiple of four bins, on both sides of one tensor box, and
    volumes that do not start on 16 bytes, against the oracle's projection."""
    from oracle import projection

    st, op = _make(nx=nx, nz=nz, n_angles=7, S=16, P=40)
    x = np.random.default_rng(8).standard_normal((nz, nx, nx)).astype(np.float32)
    buf = torch.zeros(x.size + 4, device="cuda")
    vol = buf[off:off + x.size].view(x.shape)
    vol.copy_(torch.from_numpy(x))
    assert rel_l2(_n(op.project(vol)), projection.project(x, st.angles)) < OP_TOL
    op.close()


# the tensor PSF by frequencies along z: each tile height of the batched products (rows twice
# the angles), odd and even slice counts, both trajectories and one, odd rows of bins
TENSOR = {
    "two slices": dict(nx=21, nz=2, n_angles=3, S=16, P=40, k_max=3, half_width=1),
    "odd slices, 20 rows": dict(nx=18, nz=129, n_angles=10, S=20, P=40, k_max=8, half_width=3),
    "40 rows": dict(nx=16, nz=128, n_angles=20, S=20, P=40, k_max=8, half_width=3),
    "56 rows, one trajectory": dict(nx=17, nz=130, n_angles=28, zigzag=0, S=40, P=40, k_max=18, half_width=3),
    "64 rows": dict(nx=16, nz=121, n_angles=31, S=20, P=40, k_max=8, half_width=3),
    "72 rows": dict(nx=33, nz=128, n_angles=36, S=20, P=40, k_max=8, half_width=3),
}


@pytest.mark.parametrize("name", list(TENSOR))
def test_tensor_psf_by_frequencies(name):
    from oracle import tensor_psf

    st, op = _make(**TENSOR[name])
    op.set_path("full_gemm")
    op.set_psf_model("tensor")
    rng = np.random.default_rng(9)
    gains = np.linspace(0.9, 1.1, st.n_angles)
    op.set_gain(gains.astype(np.float32))
    coil = rng.uniform(0.5, 1.5, (st.nz, st.nx)).astype(np.float32)
    x = rng.standard_normal((st.nz, st.nx, st.nx)).astype(np.float32)
    m = np.array([st.n_angles - 1])
    y = np.zeros(st.data_shape, dtype=np.complex64)
    y[m] = rng.standard_normal(y[m].shape) + 1j * rng.standard_normal(y[m].shape)
    for c in (None, coil):
        op.set_coil_map(c)
        ref = tensor_psf.forward_stages(x, st, c, angles=m)["data"][0] * gains[m[0]]
        assert rel_l2(_n(op.forward(_t(x)))[m[0]], to_interleaved(ref)) < OP_TOL
        buf = torch.zeros(2 * y.size + 4, device="cuda")  # data that do not start on 16 bytes
        yt = buf[1:1 + 2 * y.size].view(op.data_shape)
        yt.copy_(_t(to_interleaved(y)))
        ref = tensor_psf.adjoint_stages(y[m], st, c, angles=m)["vol"] * gains[m[0]]
        assert rel_l2(_n(op.adjoint(yt)), ref) < OP_TOL
    op.close()


def test_tensor_tables_follow_a_width_set_under_the_other_model():
    """The tables of the width in force, also when it was set while the collinear PSF was
    selected or the path changed meanwhile."""
    from oracle import tensor_psf

    kw = dict(nx=20, nz=6, n_angles=3, S=16, P=40, k_max=3, half_width=1)
    _, op = _make(**kw)
    op.set_path("line_gemm")
    op.set_psf_model("tensor")
    op.set_psf_model("collinear")
    op.set_fwhm(3.5)
    op.set_psf_model("tensor")
    st, _ = _make(**dict(kw, fwhm=3.5))
    x = np.random.default_rng(10).standard_normal((st.nz, st.nx, st.nx)).astype(np.float32)
    ref = to_interleaved(tensor_psf.forward(x, st))
    assert rel_l2(_n(op.forward(_t(x))), ref) < OP_TOL
    op.set_path("full_gemm")
    assert rel_l2(_n(op.forward(_t(x))), ref) < OP_TOL
    op.close()


@pytest.mark.parametrize("nx,nz,M", [(20, 5, 1), (184, 10, 11), (64, 16, 21), (184, 16, 14), (300, 16, 20)])
def test_psf_stage_of_few_lines(nx, nz, M):
    """H and its transpose where a line's outputs are spread over several blocks, with the small
    and the large register tiles, odd numbers of lines and of blocks of outputs."""
    st, op = _make(nx=nx, nz=nz, n_angles=M, S=12, P=20, Q=8)
    h = operator.psf.h((np.arange(st.n_fine)[:, None] - st.D) / st.Q - np.arange(nx)[None, :], st.fwhm)
    rng = np.random.default_rng(11)
    p = rng.standard_normal((M, nz, nx)).astype(np.float32)
    assert rel_l2(_n(op.apply_stage(1, _t(p))), p @ h.T) < OP_TOL
    f = rng.standard_normal((M, nz, st.n_fine)).astype(np.float32)
    assert rel_l2(_n(op.apply_stage(1, _t(f), transpose=True)), f @ h) < OP_TOL
    op.close()
