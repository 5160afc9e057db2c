"""Arguments of the differentiable operator that are refused before any kernel runs."""

import pytest

torch = pytest.importorskip("torch")

from paper_2511_06627_gb300.autograd import apply_a  # noqa: E402


class _NoCalls:
    """An operator that must not be reached."""

    fwhm = 2.0

    def __getattr__(self, name):
        raise AssertionError(f"{name} was called")


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_an_empty_width_is_refused(dtype):
    """With a width of no elements the last gain would pass for it."""
    with pytest.raises(IndexError):
        apply_a(_NoCalls(), torch.zeros(2, 4, 4), torch.ones(3), torch.empty(0, dtype=dtype))
