"""Calls captured into a CUDA graph after the preparation that a program makes outside of it."""

import pytest

from _helpers import ensure_library, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GEOM = dict(nx=33, nz=7, n_angles=5, S=16, P=40, A=4.0, phi0=0.2, zigzag=1, Q=4, fwhm=2.5, k_min=1, k_max=4,
            half_width=1)
SAMPLED = dict(GEOM, nx=40, S=32, P=6)
SAME = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_library()


def _captured(call):
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        out = call()
    for o in out:
        o.fill_(float("nan"))  # the graph alone has to fill it

    def replay():
        graph.replay()
        torch.cuda.synchronize()
        return [o.clone() for o in out]

    return replay


def _data(op):
    g = torch.Generator(device="cuda").manual_seed(61)
    return (torch.rand(op.vol_shape, device="cuda", generator=g), torch.randn(op.data_shape, device="cuda", generator=g))


@pytest.mark.parametrize("scans", ["z", "xz"])
@pytest.mark.parametrize("geom", [GEOM, SAMPLED], ids=["folded", "sampled"])
def test_z_drive_after_selecting_the_scan(geom, scans):
    from paper_2511_06627_gb300 import FFLOperator

    op = FFLOperator(**geom)
    x, y = _data(op)
    op.set_scans(scans)
    b, v = op.new_data(), op.new_volume()
    got = _captured(lambda: [op.forward_zdrive(x, out=b), op.adjoint_zdrive(y, out=v)])()
    assert all(torch.equal(a, c) for a, c in zip(got, (op.forward_zdrive(x), op.adjoint_zdrive(y))))
    op.close()


def test_gradients_after_a_forward_on_the_staged_path():
    """The width's operand is folded inside the graph; a replay after a new width uses that one."""
    from paper_2511_06627_gb300 import FFLOperator

    op = FFLOperator(**GEOM)
    x, y = _data(op)
    op.forward(x)
    replay = _captured(lambda: list(op.param_grad(x, y)))
    for fwhm in (2.5, 3.25):
        op.set_fwhm(fwhm)
        got = replay()
        other = FFLOperator(**dict(GEOM, fwhm=fwhm))
        for a, c in zip(got, other.param_grad(x, y)):
            assert rel_l2(a.cpu().numpy().reshape(-1), c.cpu().numpy().reshape(-1)) < SAME
        other.close()
    for a, c in zip(replay(), op.param_grad(x, y)):
        assert torch.equal(a, c)
    op.close()


def test_staged_pair_after_a_width_set_under_another_path():
    from paper_2511_06627_gb300 import FFLOperator

    op = FFLOperator(**GEOM)
    x, y = _data(op)
    op.forward(x), op.adjoint(y)
    op.set_path("line_gemm")
    op.set_fwhm(3.25)
    op.set_path("staged")
    b, v = op.new_data(), op.new_volume()
    replay = _captured(lambda: [op.forward(x, out=b), op.adjoint(y, out=v)])
    for fwhm in (3.25, 2.75):
        op.set_fwhm(fwhm)
        other = FFLOperator(**dict(GEOM, fwhm=fwhm))
        for a, c in zip(replay(), (other.forward(x), other.adjoint(y))):
            assert torch.equal(a, c)
        other.close()
    op.close()
