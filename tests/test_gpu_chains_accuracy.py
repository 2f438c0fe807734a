"""Which FP32 applications mix by register chains by default: those whose chains lose nothing against the dense form."""

import numpy as np
import pytest

from _util import make_pair, rel, to_gpu, to_np
from paper_2602_14454_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_ok):
    from paper_2602_14454_gb300 import build
    build.build()


# kappa = (1 - 2.2 c) / (1 + 2.2 b): inside 0.5, on both sides of it, beyond, and near the limit of the structured form
@pytest.mark.parametrize("Ls", [12, 16])
@pytest.mark.parametrize("b,c,chains", [(1.0, 0.0, True), (1.0, 1.0, True), (0.47, 0.0, True), (0.44, 0.0, False),
                                        (0.16, 0.0, False), (0.14, 0.0, False), (0.03, 0.0, False), (0.1, 0.97, False)])
def test_default_mixing(Ls, b, c, chains):
    dims = (4, 4, 4, 6)
    op, ref = make_pair(dims, Ls, 1.8, 0.03, b, c, "standard", 1.0, seed=3)
    x = to_gpu(ref.to_eo(inputs.gaussian_5d(dims, Ls, 5), 0))
    for dag in (False, True):
        want = ref.d_pc(x.cpu().numpy(), dag=dag)
        got = to_np(op.apply(x, op="eo", prec="f32", dag=dag))
        op.set_mix_mode("f32", 0)
        dense = to_np(op.apply(x, op="eo", prec="f32", dag=dag))
        op.set_mix_mode("f32", -1)
        assert np.array_equal(got, dense) != chains
        # both sum the same hops; 5 %: two samples of the same kind of rounding error, 10^5 entries each
        assert rel(got, want) <= 1.05 * rel(dense, want)
