"""launch_count counts every kernel of a call, as the CUDA profiling interface sees them."""

import pytest

from _helpers import ensure_library

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the z-drive's products whole, with an odd detector for the tensor PSF's padded rows; and in halves,
# with the last product of the adjoint in parts
WHOLE = dict(nx=33, nz=7, n_angles=5, S=16, P=40, A=4.0, phi0=0.2, zigzag=1, Q=4, fwhm=2.5, k_min=1, k_max=4,
             half_width=1)
HALVES = dict(WHOLE, nx=23, nz=95, n_angles=64, S=64, P=30, k_max=5)


@pytest.fixture(scope="module", autouse=True)
def _records():
    """The first session of the profiling interface in a process may miss its kernels."""
    ensure_library()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]):
        torch.ones(8, device="cuda").sum()
        torch.cuda.synchronize()


@pytest.mark.parametrize("what", ["staged", "full_gemm", "z-drive", "tensor", "tensor and coil"])
@pytest.mark.parametrize("geom", [WHOLE, HALVES], ids=["whole", "halves"])
def test_every_kernel_is_counted(geom, what):
    from paper_2511_06627_gb300 import FFLOperator

    op = FFLOperator(**geom)
    x = torch.rand(op.vol_shape, device="cuda")
    y = torch.randn(op.data_shape, device="cuda")
    b, v = op.new_data(), op.new_volume()
    if what != "z-drive" and what != "staged":
        op.set_path("full_gemm")
    if what.startswith("tensor"):
        op.set_psf_model("tensor")
    if what == "tensor and coil":
        op.set_coil_map(torch.full((op.nz, op.nx), 0.5).numpy())

    def pair():
        if what == "z-drive":
            op.forward_zdrive(x, out=b), op.adjoint_zdrive(y, out=v)
        else:
            op.forward(x, out=b), op.adjoint(y, out=v)

    pair()
    torch.cuda.synchronize()
    before = op.launch_count()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        pair()
        torch.cuda.synchronize()
    kernels = [e.name for e in prof.events() if "mpiffl" in e.name]
    if not kernels:
        pytest.skip("no kernel records from the profiling interface")
    assert op.launch_count() - before == len(kernels), kernels
    op.close()
