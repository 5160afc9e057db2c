"""The folded line stages' transposes are as near to 64 bits as the separate stages they stand for."""

import numpy as np
import pytest

from _helpers import ensure_library, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Setup, operator  # noqa: E402

SCANS = {
    "tiny": dict(nx=32, nz=16, n_angles=8, S=64, P=128, A=6.0, phi0=0.0, zigzag=1, Q=8, fwhm=2.0, k_min=1, k_max=8,
                 half_width=2),
    "small": dict(nx=64, nz=32, n_angles=6, S=64, P=192, A=6.0, phi0=0.0, zigzag=1, Q=8, fwhm=2.5, k_min=1, k_max=10,
                  half_width=2),
    "ragged": dict(nx=51, nz=19, n_angles=7, S=50, P=102, A=6.0, phi0=0.0, zigzag=1, Q=8, fwhm=2.5, k_min=1, k_max=10,
                   half_width=2),
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_library()


def _noise(op, st, seed):
    y = np.random.default_rng(seed).standard_normal(st.data_shape + (2,)).astype(np.float32)
    return y[..., 0].astype(np.complex128) + 1j * y[..., 1], torch.from_numpy(y).cuda()


# the errors of one form differ by some 5% from input to input
@pytest.mark.parametrize("name", list(SCANS))
def test_staged_adjoint_against_the_separate_stages(name):
    from paper_2511_06627_gb300 import FFLOperator

    st, op = Setup(**SCANS[name]), FFLOperator(**SCANS[name])
    yc, y = _noise(op, st, 83)
    ref = operator.adjoint(yc, st)
    stages = y
    for s in (3, 2, 1, 0):
        stages = op.apply_stage(s, stages, transpose=True)
    folded, stages = rel_l2(op.adjoint(y).cpu().numpy(), ref), rel_l2(stages.cpu().numpy(), ref)
    assert folded < 1.1 * stages, (folded, stages)
    op.close()


# plain sums of the last product were at 1.4 to 1.6 times; one trajectory, and the products in halves
ZDRIVE = dict(SCANS, **{
    "one trajectory": dict(SCANS["small"], zigzag=0),
    "halves": dict(nx=23, nz=95, n_angles=64, S=64, P=30, A=4.0, phi0=0.2, zigzag=1, Q=4, fwhm=2.5, k_min=1, k_max=5,
                   half_width=1),
})


@pytest.mark.parametrize("name", list(ZDRIVE))
def test_zdrive_adjoint_against_the_sampled_stages(name):
    from paper_2511_06627_gb300 import FFLOperator

    from oracle import zdrive

    st, op = Setup(**ZDRIVE[name]), FFLOperator(**ZDRIVE[name])
    yc, y = _noise(op, st, 84)
    m = np.arange(min(st.n_angles, 8))  # data of the other angles are zero
    yc[len(m):] = 0
    y[len(m):] = 0
    ref = zdrive.adjoint_stages_z(yc[m], st, angles=m)["vol"]
    stages = op.apply_stage_zdrive(2, op.apply_stage(3, y, transpose=True), transpose=True)
    stages = op.apply_stage(0, op.apply_stage_zdrive(1, stages, transpose=True), transpose=True)
    folded, stages = rel_l2(op.adjoint_zdrive(y).cpu().numpy(), ref), rel_l2(stages.cpu().numpy(), ref)
    assert folded < 1.2 * stages, (folded, stages)
    op.close()
