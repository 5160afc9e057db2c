"""A new PSF width reaches every path, scan and PSF model of a handle, also when an allocation
fails while its tables are rebuilt."""

import numpy as np
import pytest

from _helpers import ensure_library, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GEOM = dict(nx=33, nz=7, n_angles=5, S=16, P=40, A=4.0, phi0=0.2, zigzag=1, Q=4, fwhm=2.5, k_min=1, k_max=4,
            half_width=1)
SAME = 1e-5  # two FP32 evaluations of one operator; widths of 2.5 and 3.25 differ by percents


@pytest.fixture(scope="module")
def env():
    ensure_library()
    from paper_2511_06627_gb300 import FFLOperator
    from paper_2511_06627_gb300 import _lib as L

    x = torch.from_numpy(np.random.default_rng(21).random((GEOM["nz"], GEOM["nx"], GEOM["nx"]), dtype=np.float32)).cuda()
    refs = {}
    for w in (2.5, 3.25):
        op = FFLOperator(**dict(GEOM, fwhm=w))
        refs[w] = _outputs(op, x)
        op.close()
    yield dict(L=L, lib=L.load(), x=x, refs=refs, make=lambda: FFLOperator(**GEOM))
    L.load().mpi_ffl_test_fail_alloc(0)


def _outputs(op, x, order=("zdrive", "staged", "line_gemm", "full_gemm", "tensor")):
    """Every evaluation of the handle: the z-drive scan, each path, the tensor PSF."""
    out = {}
    for k in order:
        if k == "zdrive":
            out[k] = op.forward_zdrive(x)
            continue
        if k == "tensor":
            op.set_psf_model("tensor")
        else:
            op.set_psf_model("collinear")
            op.set_path(k)
        out[k] = op.forward(x)
        if k == "staged":
            out["width gradient"] = op.param_grad(x, out[k])[1].reshape(1)
    op.set_psf_model("collinear")
    op.sync_check()
    return {k: v.double().cpu().numpy() for k, v in out.items()}


def _agree(got, ref):
    for k, v in got.items():
        assert rel_l2(v, ref[k]) < SAME, (k, rel_l2(v, ref[k]))


def test_the_two_widths_are_told_apart(env):
    a, b = env["refs"][2.5], env["refs"][3.25]
    assert all(rel_l2(a[k], b[k]) > 100 * SAME for k in a)


@pytest.mark.parametrize("model", ["collinear", "tensor"])
@pytest.mark.parametrize("path", ["staged", "line_gemm", "full_gemm"])
def test_one_width_after_a_failed_allocation(env, path, model):
    from paper_2511_06627_gb300 import MpiFflError

    L, lib, x = env["L"], env["lib"], env["x"]
    for n in range(1, 60):
        op = env["make"]()
        _outputs(op, x)  # every table is built, for the first width
        op.set_path(path)
        op.set_psf_model(model)
        assert lib.mpi_ffl_test_fail_alloc(n) == L.OK
        failed = False
        try:
            op.set_fwhm(3.25)
        except MpiFflError as e:
            assert e.code == L.ERR_OOM, e
            failed = True
        lib.mpi_ffl_test_fail_alloc(0)
        ref = env["refs"][op.fwhm]
        _agree({"zdrive": op.forward_zdrive(x).double().cpu().numpy()}, ref)
        if not failed:
            assert op.fwhm == 3.25
            _agree({path if model == "collinear" else "tensor": op.forward(x).double().cpu().numpy()}, ref)
        _agree(_outputs(op, x), ref)
        op.close()
        if not failed:
            break
    else:
        raise AssertionError("every allocation failed")


@pytest.mark.parametrize("path", ["staged", "line_gemm", "full_gemm"])
def test_an_invalid_width_changes_nothing(env, path):
    from paper_2511_06627_gb300 import MpiFflError

    op = env["make"]()
    op.set_path(path)
    with pytest.raises(MpiFflError):
        op.set_fwhm(-1.0)
    assert op.fwhm == 2.5
    _agree(_outputs(op, env["x"]), env["refs"][2.5])
    op.close()
