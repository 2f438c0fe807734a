"""A solve follows the handle's settings of the moment, also where an earlier solve left its captured iteration."""

import numpy as np
import pytest

from _util import make_pair, to_gpu, to_np
from paper_2602_14454_gb300 import inputs

pytestmark = pytest.mark.gpu

SETTINGS = {
    "dense mixing": lambda op, prec: op.set_mix_mode(prec, 0),
    "default mixing": lambda op, prec: op.set_mix_mode(prec, -1),
    "columns of two planes": lambda op, prec: op.set_sweep(prec, 2),
    "index order": lambda op, prec: op.set_sweep(prec, 0),
}


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_ok):
    from paper_2602_14454_gb300 import build
    build.build()


# the FP32 default mixes by chains at Ls 16, which an explicit dense mode does not; a sweep changes the order of the
# norms' partial sums (by last bits that FP64 iterations keep).  Solves are reproducible bit for bit, so equality
# with a fresh handle is exact.
@pytest.mark.parametrize("first,then", [(None, "dense mixing"), ("dense mixing", "default mixing"),
                                        (None, "columns of two planes"), ("columns of two planes", "index order")])
@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_settings_after_a_solve(prec, first, then):
    dims, Ls = (8, 8, 8, 4), 16
    U = inputs.random_links(dims, 0.3, 4)
    new = lambda: make_pair(dims, Ls, 1.8, 0.1, 1.5, 0.5, "neff", 0.6, U=U)[0]
    op, fresh = new(), new()
    b5 = op.source_5d(to_gpu(inputs.gaussian_4d(dims, 6)))
    if prec == "f64":
        for o in (op, fresh):
            o.set_hop_config(prec, 0, 1, 4)
    if first:
        SETTINGS[first](op, prec)
    op.solve(b5, inner_prec=prec, tol=1e-8)
    for o in (op, fresh):
        SETTINGS[then](o, prec)
    got, want = (to_np(o.solve(b5, inner_prec=prec, tol=1e-8)[0]) for o in (op, fresh))
    assert np.array_equal(got, want)
