"""The fixed-point FP64 operator (the FP64 default) against the FP64 hop (variant 0).

Both evaluate the same sums; FP64 rounds every operation (about 60 along the
longest chain of one output, 60 * 2^-53 = 7e-15 of the largest terms), the
fixed-point form a few times at 2^-57: 1e-14 of the vector's norm bounds the
difference of the two.
"""

import numpy as np
import pytest

from _util import make_pair, rel, to_gpu, to_np
from paper_2602_14454_gb300 import inputs

pytestmark = pytest.mark.gpu
BOUND = 1e-14


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_ok):
    from paper_2602_14454_gb300 import build
    build.build()


def both(op, x, which, dag):
    """(fixed-point, FP64 variant 0) results of one application."""
    fx = to_np(op.apply(x, op=which, prec="f64", dag=dag))
    op.set_hop_config("f64", 0, 0, 0)
    ref = to_np(op.apply(x, op=which, prec="f64", dag=dag))
    op.set_hop_config("f64", -1, 0, 0)
    return fx, ref


def field(dims, Ls, which, seed):
    x = inputs.gaussian_5d(dims, Ls, seed)
    return x if which == "full" else x.reshape(Ls, -1, 4, 3)[:, ::2].copy()


# Ls: the smallest and largest, both sides of the 58/57-bit tiles, the ones with kernels of their own,
# CTAs of 128 and of fewer threads; lattices whose last CTA is full, partial and the only one
@pytest.mark.parametrize("dims,Ls", [((2, 2, 2, 2), 2), ((2, 2, 4, 6), 3), ((4, 4, 4, 4), 8), ((4, 2, 2, 6), 12),
                                     ((6, 2, 4, 2), 15), ((4, 4, 2, 4), 16), ((2, 4, 2, 4), 17), ((2, 2, 2, 10), 32)])
@pytest.mark.parametrize("b,c,form", [(1.5, 0.5, "neff"), (1.0, 0.0, "standard"), (1.0, 1.0, "standard")])
def test_matches_fp64(dims, Ls, b, c, form):
    op, _ = make_pair(dims, Ls, 1.8, 0.03, b, c, form, 0.6, seed=3)
    for which in ("eo", "full"):
        x = to_gpu(field(dims, Ls, which, 5))
        for dag in (False, True):
            fx, ref = both(op, x, which, dag)
            assert rel(fx, ref) < BOUND, (which, dag, rel(fx, ref))


@pytest.mark.parametrize("Ls", [5, 16, 20])
def test_wide_exponents(Ls):
    """Sites, slices and chiralities of very different size, zeros, and powers of two."""
    dims = (4, 4, 2, 4)
    op, _ = make_pair(dims, Ls, 1.8, 0.03, 1.5, 0.5, "neff", 0.6, seed=3)
    rng = np.random.default_rng(1)
    x = field(dims, Ls, "eo", 7)
    x *= 2.0 ** rng.integers(-60, 60, x.shape[:2] + (1, 1))
    x[:, ::5] = 0
    x[1, :, 2:] *= 1e-9
    for dag in (False, True):
        fx, ref = both(op, to_gpu(x), "eo", dag)
        # against the largest input that reaches an output: the absolute operator is below 8 neighbours
        # x sum |M| < 64 of it (two hops and two mixings), and every site reaches every other here
        assert np.abs(fx - ref).max() < 64 * 2.0 ** -53 * 8 * np.abs(x).max()
        assert rel(fx, ref) < BOUND
        for k in (-300, 400):   # exact under powers of two
            got = to_np(op.apply(to_gpu(x * 2.0 ** k), op="eo", prec="f64", dag=dag))
            assert np.array_equal(got, fx * 2.0 ** k)


def test_point_source_and_decay():
    """A single entry, and slices that fall off as a domain-wall mode does: every slice as accurate as in FP64."""
    dims, Ls = (4, 4, 4, 4), 16
    op, ref = make_pair(dims, Ls, 1.8, 0.03, 1.5, 0.5, "standard", 1.0, seed=3)
    x = np.zeros((Ls,) + ref.site_shape + (4, 3), dtype=np.complex128)
    x[3, 1, 2, 3, 0, 2, 1] = 1e-7
    fx, want = both(op, to_gpu(x), "full", False)
    assert rel(fx, want) < BOUND and np.array_equal(fx == 0, want == 0)
    x = inputs.gaussian_5d(dims, Ls, 9) * (10.0 ** -np.arange(Ls))[:, None, None, None, None, None, None]
    fx, want = both(op, to_gpu(x), "full", False)
    for s in range(Ls):
        assert rel(fx[s], want[s]) < BOUND * 10, s   # row s also takes row s - 1, ten times larger


@pytest.mark.parametrize("Ls", [8, 6])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_non_finite_values_spread_as_in_fp64(Ls, value):
    dims = (4, 4, 4, 4)
    op, _ = make_pair(dims, Ls, 1.8, 0.03, 1.5, 0.5, "standard", 1.0, seed=3)
    for which in ("eo", "full"):
        for dag in (False, True):
            x = field(dims, Ls, which, 5)
            x.reshape(-1)[x.size // 3] = value
            fx, ref = both(op, to_gpu(x), which, dag)
            ok = np.isfinite(ref)
            assert np.array_equal(np.isfinite(fx), ok) and 0 < ok.sum() < ok.size
            assert rel(fx[ok], ref[ok]) < BOUND


def test_links_outside_su3():
    """Links of any scale, zero links and a non-finite one."""
    dims, Ls = (4, 4, 4, 4), 8
    U = inputs.random_links(dims, 0.5, 3)
    rng = np.random.default_rng(2)
    U *= 2.0 ** rng.integers(-20, 20, U.shape[:-2] + (1, 1))
    U[:, 0, 1] = 0
    op, _ = make_pair(dims, Ls, 1.8, 0.03, 1.5, 0.5, "standard", 1.0, U=U)
    x = to_gpu(field(dims, Ls, "full", 5))
    fx, ref = both(op, x, "full", False)
    assert rel(fx, ref) < BOUND
    U[2, 1, 1, 2, 3, 0, 1] = np.inf
    op.set_gauge(to_gpu(U))
    fx, ref = both(op, x, "full", True)
    ok = np.isfinite(ref)
    assert np.array_equal(np.isfinite(fx), ok) and 0 < ok.sum() < ok.size
    assert rel(fx[ok], ref[ok]) < BOUND
