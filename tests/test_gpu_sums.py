"""Sums of FP32 terms with the accuracy and the range of FP64 sums: chi^2 of
wf_eval_any's mixed path and the band energies of FP32 states, for values that
grow along the map (the last terms of a sum dwarf the first) and whose squares
lie inside, above and below the FP32 range.

The terms are known exactly: with no weights chi^2 is sum w_k |s_k|^2, and at
s = 0 it is sum (w d) d with w d rounded to FP32, so Python's exact fsum of the
FP64 products is the answer.  Tolerance 1e-13: a chain of some 300 FP64 additions
of non-negative terms is within 300 x 2^-53 = 3.4e-14."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1810_00503_gb300 import synth, wf  # noqa: E402
from tests.helpers import ensure_lib, make_problem, to_dev  # noqa: E402

TOL = 1e-13
SCALES = [1e-25, 1e-18, 1.0, 1e19]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ensure_lib()


def _grow(rng, shape, scale):
    """FP32 normal deviates that grow by 1e5 along the first axis of a map."""
    ramp = np.logspace(0, 5, shape[-2])[:, None]
    return (rng.standard_normal(shape) * ramp * scale).astype(np.float32)


@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("ny,nx,C", [(7, 9, 1), (24, 30, 2), (343, 20, 1), (360, 640, 2)])
def test_chi2_of_the_mixed_any_path(ny, nx, C, scale):
    rng = np.random.default_rng(ny * nx)
    h1 = nx // 2 + 1
    P = to_dev(np.ones((C, ny, h1)), torch.float32)
    mask = rng.integers(0, 2, size=(1, ny, nx)).astype(np.uint8)
    M = to_dev(mask, torch.uint8)
    S = _grow(rng, (1, C, ny, h1), scale) + 1j * _grow(rng, (1, C, ny, h1), scale)
    zero = to_dev(np.zeros((1, C, ny, nx)), torch.float32)
    chi2, _ = wf.eval_any(to_dev(S, torch.complex64), M, zero, P, d=zero)
    w = np.full(h1, 2.0)
    w[0] = 1.0
    if nx % 2 == 0:
        w[-1] = 1.0
    sq = S.real.astype(np.float64) ** 2 + S.imag.astype(np.float64) ** 2
    ref = math.fsum((sq * w).ravel())
    assert abs(chi2.item() - ref) <= TOL * ref
    # the data term, at s = 0
    d = _grow(rng, (1, C, ny, nx), scale)
    N = rng.uniform(0.5, 1.5, size=d.shape).astype(np.float32)
    chi2, _ = wf.eval_any(torch.zeros((1, C, ny, h1), dtype=torch.complex64, device="cuda"), M, to_dev(N, torch.float32),
                          P, d=to_dev(d, torch.float32))
    wd = (N * d * mask[:, None]).astype(np.float64)
    ref = math.fsum((wd * d).ravel())
    assert abs(chi2.item() - ref) <= TOL * ref


@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("ny,nx,C", [(16, 1024, 2), (256, 64, 1)])
def test_band_energies_of_fp32_states(ny, nx, C, scale):
    rng = np.random.default_rng(ny + nx)
    inp = synth.density_small(ny, seed=1, nx=nx) if C == 1 else synth.shear_eb(ny, seed=1, nx=nx)
    prob, _ = make_problem([inp], "mixed")
    h1, nb = nx // 2 + 1, 7
    S = _grow(rng, (1, C, ny, h1), scale) + 1j * _grow(rng, (1, C, ny, h1), scale)
    band = np.sort(rng.integers(0, nb, size=(C, ny, h1)), axis=1).astype(np.int16)  # long runs of one band
    E = prob.band_energy(to_dev(S, torch.complex64), to_dev(band, torch.int16),
                         to_dev(np.full(nb, 0.5), torch.float64)).cpu().numpy()[0]
    w = np.full(h1, 2.0)
    w[0] = w[-1] = 1.0
    sq = (S[0].real.astype(np.float64) ** 2 + S[0].imag.astype(np.float64) ** 2) * w
    for l in range(nb):
        ref = math.fsum(sq[band == l])
        assert abs(E[l] - ref) <= TOL * ref
    prob.close()
