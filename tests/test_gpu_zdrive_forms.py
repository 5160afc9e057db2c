"""Forms of the z-drive scan's tables and kernels beside the ordinary ones."""

import ctypes as C
import threading

import numpy as np
import pytest

from _helpers import OP_TOL, ensure_library, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Setup, zdrive  # noqa: E402
from oracle.data import to_interleaved  # noqa: E402

GEOM = dict(nx=21, nz=9, n_angles=3, S=16, P=30, A=4.0, phi0=0.0, zigzag=1, Q=8, fwhm=2.5, k_min=1, k_max=5,
            half_width=1)
FORMS = {"folded": GEOM, "sampled": dict(GEOM, nx=40, nz=8, S=32, P=6)}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_library()


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _check(op, st):
    """A_z and A_z^T of one angle against the oracle."""
    rng = np.random.default_rng(31)
    m = np.array([st.n_angles - 1])
    x = rng.standard_normal((st.nz, st.nx, st.nx)).astype(np.float32)
    y = np.zeros(st.data_shape, dtype=np.complex64)
    y[m] = rng.standard_normal(y[m].shape) + 1j * rng.standard_normal(y[m].shape)
    b = op.forward_zdrive(_t(x)).double().cpu().numpy()
    xa = op.adjoint_zdrive(_t(to_interleaved(y))).double().cpu().numpy()
    op.sync_check()
    assert rel_l2(b[m], to_interleaved(zdrive.forward_stages_z(x, st, angles=m)["data"])) < OP_TOL
    assert rel_l2(xa, zdrive.adjoint_stages_z(y[m], st, angles=m)["vol"]) < OP_TOL


@pytest.mark.parametrize("form", list(FORMS))
def test_a_drive_amplitude_just_above_whole_fine_cells(form):
    """Q A = 24 + 4e-15 still has a margin of 24 cells; where the sine is -1 the offset must not
    fall to the cell below the first one. (The oracle takes A = 3, which differs by 4e-16.)"""
    from paper_2511_06627_gb300 import FFLOperator

    amp = (0.1 + 0.2) * 10
    assert 8 * amp > 24 and np.ceil(8 * amp - 1e-9) == 24
    op = FFLOperator(**dict(FORMS[form], A=amp))
    _check(op, Setup(**dict(FORMS[form], A=3.0)))
    op.close()


def test_without_memory_for_the_tables_the_sampled_kernels_serve():
    """An allocation of the folded form that fails leaves the scan to the sample-by-sample
    kernels, in both directions and at another width."""
    from paper_2511_06627_gb300 import FFLOperator, MpiFflError
    from paper_2511_06627_gb300 import _lib as L

    lib = L.load()
    served = 0
    for n in range(1, 40):
        op = FFLOperator(**GEOM)
        x = torch.zeros(op.vol_shape, device="cuda")
        assert lib.mpi_ffl_test_fail_alloc(n) == L.OK
        try:
            op.forward_zdrive(x)
            served += 1
            failed = False
        except MpiFflError as e:
            assert e.code == L.ERR_OOM, e
            failed = True
        lib.mpi_ffl_test_fail_alloc(0)
        for fwhm in () if failed else (2.5, 3.25):
            op.set_fwhm(fwhm)
            _check(op, Setup(**dict(GEOM, fwhm=fwhm)))
        op.close()
    assert served >= 25  # the others fell on tables that both forms need


def test_scans_of_different_phases_in_two_threads():
    """Two handles whose convolutions are one kernel with different amounts of shared memory,
    each in its own thread and stream."""
    from paper_2511_06627_gb300 import FFLOperator

    ops = [FFLOperator(**dict(GEOM, nx=40, nz=24, P=40, k_max=3, half_width=4, S=S)) for S in (128, 16)]
    xs = [torch.rand(op.vol_shape, device="cuda") for op in ops]
    refs = [op.forward_zdrive(x) for op, x in zip(ops, xs)]
    torch.cuda.synchronize()
    results = [None, None]

    def work(k):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                out = ops[k].new_data()
                for _ in range(1500):
                    ops[k].forward_zdrive(xs[k], out=out)
            stream.synchronize()
            results[k] = out
        except Exception as e:  # noqa: BLE001
            results[k] = e

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for got, ref in zip(results, refs):
        assert isinstance(got, torch.Tensor), got
        assert torch.equal(got, ref)
