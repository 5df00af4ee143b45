"""The register-resident FFT stages at the sizes where their tiling can go wrong,
against the FP64 oracle: tiles wider than the map (4, 8 and 16 packed columns),
warps with more sequences than the map has rows, one- and two-channel blocks,
every pair of passes, and batch sizes on both sides of the rule that narrows the
tiles (two blocks per SM).  Objective, Hessian-vector product, signal map and data
synthesis.

Tolerances as tests/test_gpu_ops.py: FP64 1e-12, mixed 2e-5 on fields (FP32 eps
6e-8 times at most 20 FFT stages and the residual's cancellation)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import wf_oracle as O  # noqa: E402
from paper_1810_00503_gb300 import synth  # noqa: E402
from tests.helpers import ensure_lib, make_problem, rel, rfft_u, to_dev  # noqa: E402

TOL = {"fp64": 1e-12, "mixed": 2e-5}

# (ny, nx, C, B): h = nx / 2 packed columns; the narrowing rule changes at
# B * tiles = 304 (tiles of 8 columns at ny = 1024, 16 at 256 and 512, 32 below)
SHAPES = [(8, 8, 2, 3), (8, 1024, 2, 1), (1024, 8, 1, 2), (16, 32, 1, 5), (32, 16, 2, 2), (64, 8, 1, 1),
          (128, 16, 2, 3), (256, 32, 1, 40), (32, 64, 2, 160), (64, 128, 1, 161), (512, 64, 2, 77), (128, 256, 1, 76),
          (64, 512, 2, 3), (512, 512, 1, 1)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ensure_lib()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ny,nx,C,B", SHAPES)
def test_stages_match_the_oracle(ny, nx, C, B, precision):
    tol = TOL[precision]
    fdt, npc = (torch.float64, np.complex128) if precision == "fp64" else (torch.float32, np.complex64)
    inp = synth.density_small(ny, seed=ny + nx, nx=nx) if C == 1 else synth.shear_eb(ny, seed=ny + nx, nx=nx)
    prob, host = make_problem([inp] * B, precision)
    fields = [synth.random_state(ny, C, seed=b, nx=nx) for b in (1, 2)]
    pick = np.arange(B) % 2  # two different maps in turn; the first and last of the batch are checked
    S = [rfft_u(f).astype(npc) for f in fields]
    zs = [np.fft.irfft2(s.astype(np.complex128), s=(ny, nx), norm="ortho") for s in S]
    s = to_dev(np.stack(S)[pick], torch.complex128 if precision == "fp64" else torch.complex64)
    z = to_dev(np.stack(fields)[pick], fdt)
    nz = to_dev(np.stack([inp.noise] * B), fdt)
    chi2, g = prob.eval(s)
    hv, x, sim = prob.hess_vec(s), prob.signal_map(s), prob.simulate(z, nz)
    torch.cuda.synchronize()
    d, W, P, mask = host["d"][0], host["W"][0], host["P"][0], host["mask"][0]
    for b in {0, B - 1}:
        zb = zs[pick[b]]
        assert abs(chi2[b].item() - O.chi2(zb, d, W, P)) <= tol * O.chi2(zb, d, W, P)
        assert rel(g[b].cpu().numpy(), rfft_u(O.grad(zb, d, W, P))) <= tol
        assert rel(hv[b].cpu().numpy(), rfft_u(O.hess_vec(zb, W, P))) <= tol
        assert rel(x[b].cpu().numpy(), O.apply_A(zb, P)) <= tol
        ref = O.synthesize_data(z[b].double().cpu().numpy(), nz[b].double().cpu().numpy(), mask, P)
        assert rel(sim[b].cpu().numpy(), ref) <= tol
    # maps of one parity are the same problem at the same state
    if B > 2:
        assert torch.equal(g[0], g[2 * ((B - 1) // 2)]) and torch.equal(x[1], x[2 * ((B - 2) // 2) + 1])
    prob.close()
