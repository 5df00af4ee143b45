"""Band sums (band energies and d chi2 / d log q) on both sides of the rule that
chooses their kernel: a bin per thread up to 96 bands, a bin per warp above, on
shapes with fewer columns than a block has threads, more rows than blocks and two
channels, against sums taken in FP64 with numpy.

Tolerances: FP64 1e-12.  FP32 states are summed with FP64 accuracy, so the energies
are within 1e-12 of the exact sums of the same FP32 values; the derivative's terms
a s are products rounded in FP32 (2^-24 each, 1e-6 of the sum of their moduli)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1810_00503_gb300 import synth  # noqa: E402
from tests.helpers import ensure_lib, make_problem, rfft_u, to_dev  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ensure_lib()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ny,nx,C,B,nb", [(8, 8, 1, 1, 1), (16, 1024, 2, 2, 95), (1024, 16, 1, 3, 96), (256, 256, 1, 2, 97),
                                          (128, 64, 2, 1, 300)])
def test_band_sums_match_numpy(ny, nx, C, B, nb, precision):
    rng = np.random.default_rng(ny + nx + nb)
    inp = synth.density_small(ny, seed=1, nx=nx) if C == 1 else synth.shear_eb(ny, seed=1, nx=nx)
    prob, _ = make_problem([inp] * B, precision)
    npc = np.complex128 if precision == "fp64" else np.complex64
    S = np.stack([rfft_u(synth.random_state(ny, C, seed=b, nx=nx)) for b in range(B)]).astype(npc)
    s = to_dev(S, torch.complex128 if precision == "fp64" else torch.complex64)
    h1 = nx // 2 + 1
    # runs of one band, single modes, modes in no band (-1) and ids beyond the last
    band = rng.integers(-1, nb + 2, size=(C, ny, h1)).astype(np.int16)
    band[:, ny // 2:] = np.sort(band[:, ny // 2:], axis=1)
    theta = rng.uniform(0.5, 2.0, size=nb)
    bt = to_dev(band, torch.int16)
    E = prob.band_energy(s, bt, to_dev(theta, torch.float64)).cpu().numpy()
    _, g, dq = prob.eval_bands(s, bt, nb)
    g, dq = g.cpu().numpy(), dq.cpu().numpy()
    w = np.full(h1, 2.0)
    w[0] = w[-1] = 1.0
    for b in range(B):
        x = S[b].astype(np.complex128)
        a = (S[b] - npc(0.5) * g[b]).astype(np.complex128)
        for l in range(nb):
            sel = (band == l) * w
            e = (np.abs(x) ** 2 * sel).sum() / (2 * theta[l])
            assert abs(E[b, l] - e) <= 1e-12 * e
            t = -(a.real * x.real + a.imag * x.imag) * sel
            assert abs(dq[b, l] - t.sum()) <= (1e-12 if precision == "fp64" else 1e-6) * np.abs(t).sum()
    prob.close()


def test_band_energy_of_values_beyond_a_float_sum():
    """Squares beyond the FP32 range, infinities and NaN reach the sums as in FP64."""
    prob, _ = make_problem([synth.density_small(16, seed=1)], "mixed")
    S = np.ones((1, 1, 16, 9), np.complex64)
    S[0, 0, 3, 2], S[0, 0, 5, 4], S[0, 0, 7, 7] = 3e25 + 1e25j, np.inf, np.nan
    band = np.zeros((1, 16, 9), np.int16)
    band[0, 5], band[0, 7] = 1, 2
    E = prob.band_energy(to_dev(S, torch.complex64), to_dev(band, torch.int16),
                         to_dev(np.ones(3), torch.float64)).cpu().numpy()[0]
    big = S[0, 0, 3, 2].astype(np.complex128)
    assert abs(E[0] - abs(big) ** 2) <= 1e-12 * abs(big) ** 2 and E[1] == np.inf and np.isnan(E[2])
    prob.close()
