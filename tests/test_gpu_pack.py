"""Packing, links and the 5D source at the sizes where their tiles end."""

import numpy as np
import pytest

from _util import make_pair, maxrel, rel, to_gpu, to_np
from paper_2602_14454_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_ok):
    from paper_2602_14454_gb300 import build
    build.build()


# A CTA takes 128 / Ls sites (whole fields: an even number of them) and 16 sites' links of one parity: last CTAs that
# are full and partial, one CTA only, rows (Lx) shorter than a CTA and longer
@pytest.mark.parametrize("dims,Ls", [((2, 2, 2, 2), 2), ((2, 2, 2, 2), 32), ((6, 2, 2, 2), 3), ((10, 2, 6, 2), 7),
                                     ((4, 6, 2, 2), 11), ((20, 2, 2, 4), 16), ((2, 14, 2, 2), 31)])
@pytest.mark.parametrize("c", [0.0, 0.5])
def test_full_field_and_source(dims, Ls, c):
    op, ref = make_pair(dims, Ls, 1.8, 0.1, 1.0, c, "standard", 1.0, seed=4, bc=(1, -1, 1, -1))
    x = inputs.gaussian_5d(dims, Ls, 5)
    want = ref.apply(x)
    # FP64: rounding of about 60 operations, 7e-15 of the norm; FP32 and FP16 as in the operator tests
    for prec, tol in (("f64", 1e-14), ("f32", 1e-5), ("f16", 3e-3)):
        got = to_np(op.apply(to_gpu(x), op="full", prec=prec))
        assert rel(got, want) < tol and maxrel(got, want) < 10 * tol, prec
    e = ref.to_eo(x, 0)
    assert rel(to_np(op.apply(to_gpu(e), op="eo", prec="f64")), ref.d_pc(e)) < 1e-13
    b4 = inputs.gaussian_4d(dims, 6)
    got = to_np(op.source_5d(to_gpu(b4)))
    want = ref.source_5d(b4)
    assert np.array_equal(got[1:-1], want[1:-1]) and not want[1:-1].any()
    if c == 0.0:   # a copy of the chiral halves
        assert np.array_equal(got, want)
    else:
        assert rel(got, want) < 1e-15   # a rounding each of hop, diagonal and sum


def test_source_with_different_wall_coefficients():
    """c_1 = 0: slice 1 is a copy; slice Ls hops with c_Ls."""
    from oracle import dwf as orc
    from paper_2602_14454_gb300 import dwf
    dims, Ls = (4, 2, 2, 6), 5
    cs = [0.0, 0.3, 0.2, 0.4, 0.7]
    U = inputs.random_links(dims, 0.5, 4)
    op = dwf.Operator(dims, Ls, 1.8, 0.1, [1.0] * Ls, cs)
    op.set_gauge(to_gpu(U))
    ref = orc.DWF(U, dims, Ls, 1.8, 0.1, [1.0] * Ls, cs)
    b4 = inputs.gaussian_4d(dims, 6)
    got, want = to_np(op.source_5d(to_gpu(b4))), ref.source_5d(b4)
    assert np.array_equal(got[0], want[0]) and rel(got[-1], want[-1]) < 1e-15


@pytest.mark.parametrize("Ls", [2, 4])
def test_batch_source_with_few_slices(Ls):
    """The batch's source scratch is larger than a 5D field at Ls < 5."""
    from paper_2602_14454_gb300 import dwf
    dims = (4, 4, 4, 4)
    ops = [make_pair(dims, Ls, 1.8, 0.1, 1.5, 0.5, "standard", 1.0, seed=4)[0] for _ in range(2)]
    b4 = [to_gpu(inputs.gaussian_4d(dims, s)) for s in (1, 2)]
    x4, stats = dwf.solve_batch(ops, b4, tol=1e-10)
    for op, b, x in zip(ops, b4, x4):
        want = op.project_4d(op.solve(op.source_5d(b), tol=1e-10)[0])
        assert rel(to_np(x), to_np(want)) < 1e-8   # both to 1e-10 of the source, times the condition
