"""The FP64 settings of a handle: what the entry points do with them."""

import numpy as np
import pytest
import torch

from _util import make_pair, rel, to_gpu, to_np
from paper_2602_14454_gb300 import dwf, inputs

pytestmark = pytest.mark.gpu
DIMS, LS = (8, 8, 4, 4), 8


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_ok):
    from paper_2602_14454_gb300 import build
    build.build()


def pair(**kw):
    op, ref = make_pair(DIMS, LS, 1.8, 0.03, 1.5, 0.5, "neff", 0.6, seed=3, **kw)
    return op, ref, to_gpu(ref.to_eo(inputs.gaussian_5d(DIMS, LS, 5), 0))


def test_reading_and_setting_back_changes_nothing():
    op, _, x = pair()
    want = to_np(op.apply(x, op="eo", prec="f64"))
    op.set_mix_mode("f64", op.mix_mode("f64"))
    assert np.array_equal(to_np(op.apply(x, op="eo", prec="f64")), want)
    op.set_hop_config("f64", *op.hop_config("f64"))
    assert np.array_equal(to_np(op.apply(x, op="eo", prec="f64")), want)
    op.set_hop_config("f64", 0, 1, 4)   # a choice of the FP64 kernels is reported as set
    assert op.hop_config("f64") == (0, 1, 4)


def test_reading_and_setting_back_with_varying_coefficients():
    """The resolved mixing mode is 0 here: the structured form needs constant coefficients."""
    b, c = np.linspace(1.0, 2.0, LS), np.linspace(0.2, 0.6, LS)
    op = dwf.Operator(DIMS, LS, 1.8, 0.05, list(b), list(c))
    op.set_gauge(to_gpu(inputs.random_links(DIMS, 0.3, 4)))
    x = to_gpu(inputs.gaussian_5d(DIMS, LS, 5))
    want = to_np(op.apply(x, op="full", prec="f64"))
    op.set_mix_mode("f64", op.mix_mode("f64"))
    assert np.array_equal(to_np(op.apply(x, op="full", prec="f64")), want)


@pytest.mark.parametrize("ns,sb", [(2, 0), (1, 8), (0, 5)])
def test_a_tile_shape_selects_the_kernels_that_take_it(ns, sb):
    op, _, x = pair()
    op.set_hop_config("f64", -1, ns, sb)
    got = to_np(op.apply(x, op="eo", prec="f64"))
    op.set_hop_config("f64", 0, ns, sb)
    assert np.array_equal(got, to_np(op.apply(x, op="eo", prec="f64")))


@pytest.mark.parametrize("Ls", [8, 10])   # 16 sites to a CTA: half a run of 32; 12 sites straddle runs (index order then)
def test_sweep_order_of_the_default(Ls):
    dims = (8, 8, 8, 4)
    op, ref = make_pair(dims, Ls, 1.8, 0.1, 1.5, 0.5, "neff", 0.6, seed=3)
    x = to_gpu(ref.to_eo(inputs.gaussian_5d(dims, Ls, 5), 0))
    b5 = op.source_5d(to_gpu(inputs.gaussian_4d(dims, 6)))
    want, x5 = to_np(op.apply(x, op="eo", prec="f64")), to_np(op.solve(b5, inner_prec="f64", tol=1e-10)[0])
    op.set_sweep("f64", 2)
    assert np.array_equal(to_np(op.apply(x, op="eo", prec="f64")), want)
    swept, st = op.solve(b5, inner_prec="f64", tol=1e-10)
    swept = to_np(swept)
    assert st["true_residual"] < 1e-10 and rel(swept, x5) < 1e-8
    # the order of the norms' partial sums, and with it the last bits, follows the sweep
    assert np.array_equal(swept, x5) == (Ls == 10)


def test_source_follows_the_choice_of_fp64_arithmetic():
    """Unit links keep colours apart: in FP64 a colour far below the others stays accurate to its own size."""
    U = np.zeros((4,) + DIMS[::-1] + (3, 3), dtype=np.complex128)
    U[..., range(3), range(3)] = 1.0
    op, ref, _ = pair(U=U)
    b4 = inputs.gaussian_4d(DIMS, 6)
    b4[..., 1] *= 2.0 ** -80
    want = ref.source_5d(b4)
    op.set_hop_config("f64", 0, 0, 0)
    got = to_np(op.source_5d(to_gpu(b4)))
    for a in range(3):   # a rounding each of eight directions' sum, diagonal and the two's sum
        assert rel(got[..., a], want[..., a]) < 1e-15, a


def test_time_mix_times_the_default():
    op, _, _ = pair()
    for mode in (-1, 0, 1):
        us, nbytes = op.time_mix("f64", mode, reps=2, flush_l2=False)
        assert us > 0 and nbytes == 2 * 24 * 8 * LS * np.prod(DIMS) / 2
    assert op.time_mix("f32", -1, reps=2, flush_l2=False)[0] > 0
    with pytest.raises(dwf.DwfError):
        op.time_mix("f64", 2, reps=2)


@pytest.mark.parametrize("prec,line", [("f64", "0 1 8 1 100.0"), ("f32", "0 1 8 0 100.0")])
def test_autotune_does_not_take_lines_of_other_kernel_sets(tmp_path, prec, line):
    """A line without the kernel set's number, as earlier libraries wrote them, is left alone."""
    op, _, _ = pair()
    cache = tmp_path / "tune.txt"
    key = "%s|%dx%dx%dx%d|Ls=%d|prec=%d" % ((torch.cuda.get_device_name().replace(" ", "_"),) + DIMS + (LS, dwf.PREC[prec]))
    cache.write_text("%s %s\n" % (key, line))
    cfg = op.autotune(prec, str(cache))
    lines = cache.read_text().splitlines()
    assert len(lines) == 2 and lines[0] == "%s %s" % (key, line) and not lines[1].startswith(key + " ")
    op2, _, _ = pair()
    assert op2.autotune(prec, str(cache)) == cfg and len(cache.read_text().splitlines()) == 2   # the new line is taken
