"""workspace_bytes is the device memory a handle holds, whatever it has built, and a request's
estimate covers what it will hold."""

import ctypes as C

import pytest

from _helpers import ensure_library

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GEOM = dict(nx=33, nz=7, n_angles=5, S=16, P=40, A=4.0, phi0=0.2, zigzag=1, Q=4, fwhm=2.5, k_min=1, k_max=4,
            half_width=1)


def _live(lib):
    n, b = C.c_int64(), C.c_int64()
    lib.mpi_ffl_test_live_allocs(C.byref(n), C.byref(b))
    return b.value


def _held(lib, L, op):
    sz = L.Sizes()
    assert lib.mpi_ffl_get_sizes(op._h, C.byref(sz)) == L.OK
    return sz.workspace_bytes


def test_workspace_bytes_after_each_first_use():
    ensure_library()
    from paper_2511_06627_gb300 import FFLOperator
    from paper_2511_06627_gb300 import _lib as L

    lib = L.load()
    base = _live(lib)
    op = FFLOperator(**GEOM)
    x = torch.rand(op.vol_shape, device="cuda")
    y = torch.randn(op.data_shape, device="cuda")
    steps = [
        lambda: None,
        lambda: op.forward(x),
        lambda: op.param_grad(x, y),
        lambda: op.forward_zdrive(x),
        lambda: op.apply_stage_zdrive(2, op.apply_stage_zdrive(1, op.apply_stage(0, x))),
        lambda: op.set_path("full_gemm"),
        lambda: op.set_psf_model("tensor"),
        lambda: op.set_fwhm(3.0),
        lambda: op.set_scans("xz"),
        lambda: op.solve(torch.cat((y, y)), iters=2, n_power=2),
        lambda: op.set_coil_map(torch.ones(op.nz, op.nx).numpy()),
        lambda: op.set_coil_map(None),
        lambda: op.forward(x.cpu().pin_memory()),
    ]
    for k, step in enumerate(steps):
        step()
        torch.cuda.synchronize()
        assert _held(lib, L, op) == _live(lib) - base, k
    op.close()
    assert _live(lib) == base


@pytest.mark.parametrize("geom", [
    GEOM,
    dict(GEOM, nx=40, nz=8, n_angles=12, S=128, P=80, A=6.0, Q=8, zigzag=0, k_min=2, k_max=8, half_width=3),
    dict(nx=64, nz=64, n_angles=12, S=64, P=192, A=6.0, Q=8, fwhm=2.5, k_min=1, k_max=8, half_width=2),
    dict(nx=128, nz=64, n_angles=24, S=64, P=256, A=6.0, Q=8, fwhm=3.0, k_min=1, k_max=12, half_width=3),
    dict(nx=256, nz=128, n_angles=36, S=128, P=512, A=6.0, Q=8, fwhm=3.0, k_min=1, k_max=16, half_width=4),
], ids=lambda g: f"{g['nx']}x{g['nz']}")
def test_a_request_holds_no_more_than_its_estimate(geom):
    ensure_library()
    from paper_2511_06627_gb300 import _lib as L
    from paper_2511_06627_gb300.serving import Job, Request, _declare, estimate_request_bytes

    lib = L.load()
    _declare(lib)
    nb = (geom["k_max"] - geom["k_min"] + 1) * (2 * geom["half_width"] + 1)
    data = torch.randn(geom["n_angles"], geom["nz"], nb, 2)
    base = _live(lib)
    job = Job(Request(geometry=geom, data=data, iters=2, n_power=2, name="r"), "full_gemm", None)
    torch.cuda.synchronize()
    held, estimate = _live(lib) - base, estimate_request_bytes(geom)
    job.release()
    assert held <= estimate
    assert estimate < 1.5 * held + (24 << 20)  # and not much more, so that the budget is used
