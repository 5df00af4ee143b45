"""Row stage of wf_eval_any on both sides of the rule that chooses it: a warp takes
a pair of rows, and a whole block where a call has too few pairs to fill the chip.
The values are the same, so a batch's gradients equal those of its maps alone bit
for bit, and chi^2 differs by the order of its sums only (1e-13, some 300 FP64
additions of non-negative terms).  Lengths of every radix and number of passes
whose widest pass is wider than a warp, with an odd last row."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1810_00503_gb300 import wf  # noqa: E402
from tests.helpers import ensure_lib  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ensure_lib()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nx", [98, 135, 243, 324, 343, 441, 625, 686, 735, 768, 875, 945, 1000, 1024])
@pytest.mark.parametrize("ny,C,B", [(5, 1, 250), (9, 2, 70), (60, 1, 11)])
def test_batch_equals_its_maps_alone(ny, nx, C, B, dtype):
    g = torch.Generator(device="cuda").manual_seed(nx + ny)
    h1 = nx // 2 + 1
    mask = (torch.rand(B, ny, nx, device="cuda", generator=g) > 0.3).to(torch.uint8)
    Ninv = torch.rand(B, C, ny, nx, dtype=dtype, device="cuda", generator=g) + 0.5
    P = torch.rand(C, ny, h1, dtype=dtype, device="cuda", generator=g)
    d = torch.randn(B, C, ny, nx, dtype=dtype, device="cuda", generator=g)
    s = torch.randn(B, C, ny, h1, 2, dtype=dtype, device="cuda", generator=g)
    s = torch.view_as_complex(s)
    chi2, grad = wf.eval_any(s, mask, Ninv, P, d=d)
    for b in (0, B - 1):
        one = slice(b, b + 1)
        c1, g1 = wf.eval_any(s[one], mask[one], Ninv[one], P, d=d[one])
        assert torch.equal(g1[0], grad[b])
        assert abs(c1.item() - chi2[b].item()) <= 1e-13 * c1.item()
