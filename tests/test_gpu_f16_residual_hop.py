"""FP16 inner iterations whose K_d runs the warp-autonomous hop (Ls 8 and 16), and one that does not (Ls 12)."""

import pytest

from _util import make_pair, to_gpu, to_np
from paper_2602_14454_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_ok):
    from paper_2602_14454_gb300 import build
    build.build()


@pytest.mark.parametrize("Ls", [8, 12, 16])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 6, 4)])
def test_solve(dims, Ls):
    op, ref = make_pair(dims, Ls, 1.8, 0.1, 1.5, 0.5, "neff", 0.6, seed=3)
    b5 = ref.source_5d(inputs.gaussian_4d(dims, 6))
    x5, st = op.solve(to_gpu(b5), inner_prec="f16", tol=1e-10)
    assert st["status"] == "DWF_OK" and ref.residual_norm(b5, to_np(x5)) < 1e-10   # the solver's own bound
    plain, st0 = op.solve(to_gpu(b5), inner_prec="f32", tol=1e-10)
    assert st["iterations"] < 3 * st0["iterations"]   # the residual hop keeps FP16's convergence
