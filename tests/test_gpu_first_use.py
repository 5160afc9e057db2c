"""Tables built on the first use of a handle: that use on a stream of its own."""

import numpy as np
import pytest

from _helpers import ensure_library

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# a small scan, whose line operator is built on the host, and one above that size
SCANS = {
    "small": dict(nx=33, nz=7, n_angles=5, S=16, P=40, A=4.0, phi0=0.2, zigzag=1, Q=4, fwhm=2.5, k_min=1, k_max=4,
                  half_width=1),
    "larger": dict(nx=72, nz=12, n_angles=6, S=64, P=128, A=6.0, phi0=0.0, zigzag=1, Q=8, fwhm=3.0, k_min=1, k_max=10,
                   half_width=2),
    "sampled z": dict(nx=40, nz=8, n_angles=3, S=32, P=6, A=4.0, phi0=0.2, zigzag=1, Q=4, fwhm=2.5, k_min=1, k_max=5,
                      half_width=1),
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_library()


def _calls(op, x, y, what):
    if what == "staged":
        return [op.forward(x), op.adjoint(y)]
    if what == "gradients":
        return list(op.param_grad(x, y))
    if what == "z-drive":
        return [op.forward_zdrive(x), op.adjoint_zdrive(y)]
    if what == "z stages":
        return [op.apply_stage_zdrive(2, op.apply_stage_zdrive(1, op.apply_stage(0, x)))]
    if what == "new gains":
        op.set_gain(np.linspace(0.9, 1.1, op.n_angles).astype(np.float32))
        return [op.forward(x), op.adjoint(y)]
    op.set_path("full_gemm")
    if what == "tensor":
        op.set_psf_model("tensor")
    return [op.forward(x), op.adjoint(y)]


@pytest.mark.parametrize("what", ["staged", "gradients", "z-drive", "z stages", "new gains", "full_gemm", "tensor"])
@pytest.mark.parametrize("scan", list(SCANS))
def test_first_use_on_a_side_stream(scan, what):
    from paper_2511_06627_gb300 import FFLOperator

    g = torch.Generator(device="cuda").manual_seed(41)
    op = FFLOperator(**SCANS[scan])
    x = torch.rand(op.vol_shape, device="cuda", generator=g)
    y = torch.randn(op.data_shape, device="cuda", generator=g)
    ref = _calls(op, x, y, what)
    torch.cuda.synchronize()
    op.close()
    for _ in range(3):
        op = FFLOperator(**SCANS[scan])
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            got = _calls(op, x, y, what)
        side.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, ref))
        op.sync_check()
        op.close()
