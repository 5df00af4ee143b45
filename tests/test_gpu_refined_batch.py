"""Certified solves (wf_map_solve_refined) of MIXED batches large enough that no
stage narrows its tiles: the FP64 outer evaluations then run the FP64 stages'
own widest tiles, which differ from the FP32 ones at sides of 32, 128 and 512.
Every map has to end where the same map ends in a batch of two.

Tolerance: a certificate of 1e-7 puts each state within 1e-7 |s| of the MAP, so
two of them are within 2e-7 of each other."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1810_00503_gb300 import synth  # noqa: E402
from tests.helpers import ensure_lib, make_problem  # noqa: E402

TOL = 1e-7


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ensure_lib()


@pytest.mark.parametrize("ny,nx,C,B", [(512, 512, 2, 20), (128, 128, 1, 160), (128, 1024, 1, 20), (1024, 512, 1, 10),
                                       (256, 32, 2, 80)])
def test_refined_mixed_batch_ends_where_a_small_batch_ends(ny, nx, C, B):
    maker = synth.density_small if C == 1 else synth.shear_eb
    pair = [maker(ny, seed=11 + i, nx=nx) for i in range(2)]
    opts = dict(cert_tol=TOL, max_rounds=8, gtol_rel=1e-6, max_iter=20000)
    out = []
    for n in (2, B):
        prob, _ = make_problem(pair * (n // 2), "mixed")
        res, cert = prob.solve_refined(**opts)
        assert {st["status"] for st in res.stats} == {"WF_OK"} and cert.max() <= TOL
        out.append(res.s)
        prob.close()
    small, s = out
    for b in range(B):
        ref = small[b % 2]
        assert torch.linalg.vector_norm(s[b] - ref) <= 2 * TOL * torch.linalg.vector_norm(ref)
