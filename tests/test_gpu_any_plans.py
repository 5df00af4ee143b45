"""Objective of wf_eval_any at side lengths that take every radix of its
transforms (2 to 16, composite ones included) and two to four passes, with an
odd number of rows (the last pair of rows has one) and column tiles with a
ragged end, against the FP64 oracle.  Tolerances: FP64 1e-12; FP32 2e-5 for the
field and 1e-5 for chi^2, the bounds of the other tests of this path."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.helpers import ensure_lib  # noqa: E402
from tests.test_gpu_any import _run  # noqa: E402

LENGTHS = [10, 14, 16, 27, 32, 35, 75, 81, 98, 112, 135, 144, 175, 243, 288, 441, 512, 625, 686, 729, 875, 900, 945,
           960, 972, 980, 1008, 1024]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ensure_lib()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("L", LENGTHS)
def test_every_radix_along_both_axes(L, precision):
    _run(L, 9, 1, 2, precision, seed=L)  # columns of L
    _run(5, L, 1, 2, precision, seed=L + 1)  # rows of L, an odd number of them
