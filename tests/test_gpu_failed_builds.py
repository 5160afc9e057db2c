"""Every device allocation of what a handle builds on first use may fail: the call reports it,
nothing of the build is kept, and the same call made again gives what it gives otherwise."""

import ctypes as C

import pytest

from _helpers import ensure_library

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GEOM = dict(nx=33, nz=7, n_angles=5, S=16, P=40, A=4.0, phi0=0.2, zigzag=1, Q=4, fwhm=2.5, k_min=1, k_max=4,
            half_width=1)
LARGER = dict(GEOM, nx=72, nz=12, S=64, P=128, Q=8, k_max=10, half_width=2)  # W is built on the device

CALLS = {
    "staged": lambda op, x, y: [op.forward(x), op.adjoint(y)],
    "gradients": lambda op, x, y: list(op.param_grad(x, y)),
    "line_gemm": lambda op, x, y: [op.set_path("line_gemm"), op.forward(x), op.adjoint(y)][1:],
    "full_gemm": lambda op, x, y: [op.set_path("full_gemm"), op.forward(x), op.adjoint(y)][1:],
    "tensor": lambda op, x, y: [op.set_psf_model("tensor"), op.forward(x), op.adjoint(y)][1:],
    "sampled z stages": lambda op, x, y: [op.apply_stage_zdrive(2, op.apply_stage_zdrive(1, op.apply_stage(0, x)))],
}


@pytest.mark.parametrize("what", list(CALLS))
@pytest.mark.parametrize("geom", [GEOM, LARGER], ids=["host W", "device W"])
def test_every_allocation_of_a_first_use_may_fail(geom, what):
    ensure_library()
    from paper_2511_06627_gb300 import FFLOperator, MpiFflError
    from paper_2511_06627_gb300 import _lib as L

    lib = L.load()

    def live():
        n, b = C.c_int64(), C.c_int64()
        lib.mpi_ffl_test_live_allocs(C.byref(n), C.byref(b))
        return n.value, b.value

    g = torch.Generator(device="cuda").manual_seed(71)
    op = FFLOperator(**geom)
    x = torch.rand(op.vol_shape, device="cuda", generator=g)
    y = torch.randn(op.data_shape, device="cuda", generator=g)
    ref = CALLS[what](op, x, y)
    op.close()
    base = live()
    failures = 0
    for n in range(1, 80):
        op = FFLOperator(**geom)
        created = live()
        assert lib.mpi_ffl_test_fail_alloc(n) == L.OK
        try:
            CALLS[what](op, x, y)
            failed = False
        except MpiFflError as e:
            assert e.code == L.ERR_OOM, (n, e)
            failed = True
        lib.mpi_ffl_test_fail_alloc(0)
        if failed:
            failures += 1
            if what != "sampled z stages":  # its tables are kept one by one
                assert live() == created, n
            for a, b in zip(CALLS[what](op, x, y), ref):
                assert torch.equal(a, b), n
        op.close()
        assert live() == base, n
        if not failed:
            break
    assert not failed and failures >= 6
