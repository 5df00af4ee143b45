"""Shared launches (wf_map_solve_many) of problems with sides of 256, 512 and
1024 along either axis, at the widest tiles (autotune off), whose row blocks need
more shared memory than any column tile; and a batch of one problem that runs its
FFT stages in launches of its own (1024 column tiles or more) beside one that
shares them.  Every map ends exactly where its problem alone ends with the same
stages: the same states bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1810_00503_gb300 import wf  # noqa: E402
from tests.helpers import ensure_lib  # noqa: E402
from tests.test_gpu_multi import SHARED_VARIANT, _problems  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ensure_lib()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("C,shapes", [
    (1, [(64, 64, 3), (512, 512, 2)]),
    (1, [(64, 64, 3), (1024, 1024, 2)]),
    (2, [(16, 512, 1), (256, 256, 2), (32, 1024, 2)]),
    (2, [(512, 16, 1), (1024, 64, 2), (1024, 1024, 1)]),
    (1, [(512, 512, 33), (128, 512, 2)]),
])
def test_shared_launches_of_long_sides(C, shapes, precision):
    opts = dict(gtol_rel=0.0, max_iter=12, check_every=4, autotune=0)
    probs = [p for p, _ in _problems(shapes, C, precision, seed=80)]
    together = wf.solve_many(probs, **opts)
    for p, r in zip(probs, together):
        assert {s["fft_variant"] for s in r.stats} == {SHARED_VARIANT}
        alone = p.solve(fft_variant=SHARED_VARIANT, **opts)
        assert torch.equal(r.s, alone.s)
        assert [s["iters"] for s in r.stats] == [s["iters"] for s in alone.stats] == [12] * len(r.stats)
        p.close()
