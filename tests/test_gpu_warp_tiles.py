"""The warp-autonomous FP32 hop where Ls does not divide 32, its chains at Ls 12, and its batched form.

Bounds: FP32 rounding, 24 bits, of about 60 + Ls operations per output, 1e-5 of the
norm as in the operator tests; solutions to 1e-10 of the source against one another.
"""

import numpy as np
import pytest

from _util import TOL, make_pair, rel, to_gpu, to_np
from paper_2602_14454_gb300 import dwf, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_ok):
    from paper_2602_14454_gb300 import build
    build.build()


# 10, 6, 5, 4, 3, 2 and 1 sites per warp tile with idle lanes; lattices that end inside a warp tile and inside a CTA
@pytest.mark.parametrize("Ls", [3, 5, 6, 7, 9, 10, 11, 13, 14, 17, 31])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 6)])
def test_any_ls(dims, Ls):
    op, ref = make_pair(dims, Ls, 1.8, 0.03, 1.5, 0.5, "neff", 0.6, seed=3)
    x = inputs.gaussian_5d(dims, Ls, 5)
    e = ref.to_eo(x, 0)
    for dag in (False, True):
        assert rel(to_np(op.apply(to_gpu(x), op="full", prec="f32", dag=dag)), ref.apply(x, dag=dag)) < TOL["f32"]
        assert rel(to_np(op.apply(to_gpu(e), op="eo", prec="f32", dag=dag)), ref.d_pc(e, dag=dag)) < TOL["f32"]


def test_columns_that_a_tile_would_straddle():
    """Ls 10: tiles of 3 sites against column runs of 32 sites; the sweep order must not change the result."""
    dims, Ls = (8, 4, 4, 4), 10
    op, ref = make_pair(dims, Ls, 1.8, 0.03, 1.5, 0.5, "neff", 0.6, seed=3)
    e = to_gpu(ref.to_eo(inputs.gaussian_5d(dims, Ls, 5), 0))
    want = to_np(op.apply(e, op="eo", prec="f32"))
    op.set_sweep("f32", 2)
    assert np.array_equal(to_np(op.apply(e, op="eo", prec="f32")), want)


@pytest.mark.parametrize("Ls", [8, 10, 12, 16])
@pytest.mark.parametrize("eo_form", [0, 1])
def test_solve(Ls, eo_form):
    dims = (4, 4, 4, 6)
    op, ref = make_pair(dims, Ls, 1.8, 0.1, 1.5, 0.5, "neff", 0.6, seed=3)
    b5 = ref.source_5d(inputs.gaussian_4d(dims, 6))
    x5, st = op.solve(to_gpu(b5), inner_prec="f32", tol=1e-10, eo_form=eo_form)
    assert st["status"] == "DWF_OK" and ref.residual_norm(b5, to_np(x5)) < 1e-10


@pytest.mark.parametrize("setup", ["default", "one on variant 0", "one with structured mixing", "no graph"])
def test_batch(setup):
    """Systems of three Ls (one without chains, one that does not divide 32), shared and own handles."""
    dims = (4, 4, 4, 6)
    U = inputs.random_links(dims, 0.3, 4)
    ops = [make_pair(dims, Ls, 1.8, mf, 1.5, 0.5, "standard", 1.0, U=U)[0] for Ls in (8, 10, 12) for mf in (0.1, 0.2)]
    if setup == "one on variant 0":
        ops[5].set_hop_config("f32", 0, 1, 4)
    if setup == "one with structured mixing":
        ops[4].set_mix_mode("f32", 1)
    ops = ops + ops[:2]
    b4 = [to_gpu(inputs.gaussian_4d(dims, s)) for s in range(len(ops))]
    x4, stats = dwf.solve_batch(ops, b4, tol=1e-10, inner_prec="f32", use_graph=int(setup != "no graph"))
    for op, b, x, st in zip(ops, b4, x4, stats):
        assert st["status"] == "DWF_OK" and st["true_residual"] < 1e-10
        want = op.project_4d(op.solve(op.source_5d(b), tol=1e-10)[0])
        assert rel(to_np(x), to_np(want)) < 1e-8
