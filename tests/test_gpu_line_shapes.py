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
