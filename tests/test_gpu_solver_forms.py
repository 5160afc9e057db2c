"""Forms of the solver's, the batch's and the gradients' kernels beside the ordinary ones: detectors
that are not a multiple of four bins or wider than the interleaved projector takes, iterates off 16
bytes, jobs of ragged and different detectors in one batch, gradients with a coil map."""

import ctypes as C

import numpy as np
import pytest

from _helpers import OP_TOL, ensure_library, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GEOM = dict(nx=32, nz=7, n_angles=5, S=16, P=40, A=4.0, phi0=0.2, zigzag=1, Q=4, fwhm=2.5, k_min=1, k_max=4,
            half_width=1)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_library()


def _op(path, **kw):
    from paper_2511_06627_gb300 import FFLOperator

    return FFLOperator(**dict(GEOM, **kw), path=path)


def _solve_at(op, b, x, iters, lam, tau):
    """mpi_ffl_solve on the volume x in place (the wrapper's own volumes start on 16 bytes)."""
    from paper_2511_06627_gb300 import _lib as L

    p = L.SolveParams(iters, lam, tau, 10, C.c_uint64(1234), 1, 0.0, 0.0)
    rc = op._lib.mpi_ffl_solve(op._h, b.data_ptr(), x.data_ptr(), C.byref(p), None,
                               torch.cuda.current_stream().cuda_stream)
    assert rc == L.OK
    torch.cuda.synchronize()
    return x


def _reference(op, b, x0, iters, lam, tau):
    """Eq. (26) in 64 bits around the operator's own products."""
    x = x0.double()
    xp = x
    for k in range(1, iters + 1):
        y = x + (k - 1) / (k + 2) * (x - xp)
        g = op.adjoint((op.forward(y.float()) - b)).double()
        ttt = torch.zeros_like(y)
        for axis in range(3):
            d = torch.diff(y, dim=axis)
            n = y.shape[axis]
            ttt.narrow(axis, 0, n - 1).sub_(d)
            ttt.narrow(axis, 1, n - 1).add_(d)
        xp, x = x, torch.clamp(y - tau * (g + lam * ttt), min=0)
    return x


# 32: both vector forms; 33: the interleaved projector's ragged copy; 500: the plain projector, whose
# extrapolation is a pass of its own; each with iterates that start on 16 bytes and that do not
@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("nx,nz,path", [(32, 7, "full_gemm"), (33, 7, "staged"), (101, 5, "line_gemm"), (500, 2, "staged")])
def test_solve_against_the_iteration_in_64_bits(nx, nz, path, off):
    op = _op(path, nx=nx, nz=nz)
    g = torch.Generator(device="cuda").manual_seed(81)
    b = op.forward(torch.rand(op.vol_shape, device="cuda", generator=g)).clone()
    ata = op.power_norm(20, 7)
    lam, tau, iters = 1e-3 * ata, 0.9 / ata, 6
    x0 = 0.1 * torch.rand(op.vol_shape, device="cuda", generator=g)
    buf = torch.zeros(x0.numel() + 4, device="cuda")
    x = buf[off:off + x0.numel()].view(x0.shape)
    x.copy_(x0)
    got = _solve_at(op, b, x, iters, lam, tau)
    ref = _reference(op, b, x0, iters, lam, tau)
    assert rel_l2(got.cpu().numpy(), ref.cpu().numpy()) < OP_TOL
    assert float(buf[:off].abs().sum()) == 0 and float(buf[off + x0.numel():].abs().sum()) == 0
    op.close()


# every pair and mix of a multiple of four, ragged detectors on both sides of a ring stride, and one
# column more than a tile of the copy
MIX = [dict(nx=32), dict(nx=33, nz=9), dict(nx=63, n_angles=4), dict(nx=66, nz=3), dict(nx=21, zigzag=0)]


@pytest.mark.parametrize("tf32", [False, True])
def test_ragged_jobs_alone_and_in_the_mix(tf32):
    from paper_2511_06627_gb300 import PREC_TF32
    from paper_2511_06627_gb300 import _lib as L

    stream = torch.cuda.current_stream().cuda_stream
    lib, iters = L.load(), 7
    problems = []
    for k, kw in enumerate(MIX):
        op = _op("full_gemm", **kw)
        if tf32:
            op.set_precision(PREC_TF32)
        g = torch.Generator(device="cuda").manual_seed(90 + k)
        b = op.forward(torch.rand(op.vol_shape, device="cuda", generator=g)).clone()
        ata = op.power_norm(20, 7)
        problems.append((op, b, 1e-3 * ata, 0.9 / ata))

    def run(members):
        jobs = []
        for op, b, lam, tau in members:
            p = L.SolveParams(iters, lam, tau, 10, C.c_uint64(1234), 1, 0.0, 0.0)
            h = C.c_void_p()
            assert lib.mpi_ffl_job_create(op._h, b.data_ptr(), None, C.byref(p), C.byref(h), stream) == L.OK
            jobs.append(h)
        arr = (C.c_void_p * len(jobs))(*[h.value for h in jobs])
        for _ in range(iters):
            assert lib.mpi_ffl_job_step(arr, len(jobs), stream) == L.OK
        out = []
        for (op, *_), h in zip(members, jobs):
            out.append(op.new_volume())
            assert lib.mpi_ffl_job_result(h, out[-1].data_ptr(), stream) == L.OK
        torch.cuda.synchronize()
        for h in jobs:
            lib.mpi_ffl_job_destroy(h)
        return out

    alone = [run([p])[0] for p in problems]
    for (op, b, lam, tau), x in zip(problems, alone):
        ref, _ = op.solve(b, iters=iters, lam=lam, tau=tau)
        assert rel_l2(x.cpu().numpy(), ref.cpu().numpy()) < OP_TOL
    for order in ([0, 1, 2, 3, 4], [4, 3, 2, 1, 0], [3, 1], [1, 4]):
        for k, x in zip(order, run([problems[k] for k in order])):
            assert torch.equal(x, alone[k]), (order, k)
    for op, *_ in problems:
        op.sync_check()
        op.close()


@pytest.mark.parametrize("nx,nz", [(32, 7), (33, 8)])
def test_gradients_with_a_coil_map_on_every_path(nx, nz):
    """Against the products they are made of: <g_b, A_m x> at unit gains, and the difference
    quotient of the staged path's forward, whose own gradient comes from another operand."""
    op = _op("staged", nx=nx, nz=nz)
    rng = np.random.default_rng(82)
    op.set_coil_map(rng.uniform(0.5, 1.5, (nz, nx)).astype(np.float32))
    gains = rng.uniform(0.8, 1.2, op.n_angles).astype(np.float32)
    op.set_gain(gains)
    x = torch.from_numpy(rng.random(op.vol_shape, dtype=np.float32)).cuda()
    h = 0.05  # the misfit of a wider scan: its inner product with dA / dfwhm does not cancel
    op.set_fwhm(2.5 + h)
    wide = op.forward(x).double()
    op.set_fwhm(2.5)
    gb = ((wide - op.forward(x).double()) / h).float()
    unit = op.forward(x).double() / torch.from_numpy(gains).cuda().view(-1, 1, 1, 1)
    ref_g = (gb.double() * unit).flatten(1).sum(1)
    scale = float((gb.double().flatten(1).norm(dim=1) * unit.flatten(1).norm(dim=1)).max())
    ref_w = float(op.param_grad(x, gb)[1])
    assert abs(ref_w / float((gb.double() ** 2).sum()) - 1) < 0.1  # the quotient's own error is of order h
    for path in ("staged", "line_gemm", "full_gemm"):
        op.set_path(path)
        gg, gw = op.param_grad(x, gb)
        assert float((gg.double() - ref_g).abs().max()) < OP_TOL * scale, path
        assert abs(float(gw) / ref_w - 1) < 4 * OP_TOL, path
    op.close()
