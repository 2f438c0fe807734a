"""Accuracy of the FP64 operator's fixed-point default, entry by entry and against extended precision."""

import numpy as np
import pytest

from _util import make_pair, to_gpu, to_np
from paper_2602_14454_gb300 import dwf, inputs

pytestmark = pytest.mark.gpu
AXIS = (3, 2, 1, 0)   # axis of (Lt, Lz, Ly, Lx) along x, y, z, t


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_ok):
    from paper_2602_14454_gb300 import build
    build.build()


def both(op, call):
    """(default, FP64 variant 0) results of call()."""
    fx = to_np(call())
    op.set_hop_config("f64", 0, 0, 0)
    ref = to_np(call())
    op.set_hop_config("f64", -1, 0, 0)
    return fx, ref


def halves(v):
    """The largest |re| or |im| of each half block (site, s, chirality), chirality first."""
    a = np.maximum(np.abs(v.real), np.abs(v.imag)).max(-1)
    return np.stack((a[..., :2].max(-1), a[..., 2:].max(-1)))


def matrices(dims, Ls, M0, mf, b, c, form, alpha):
    """|P| and |A5 R| per chirality: D x = A5 R x - 1/2 H P x."""
    op = dwf.Operator(dims, Ls, M0, mf, b, c, form=form, alpha=alpha)
    A5, B, R = ([op.fifth_matrix(w, chi) for chi in (0, 1)] for w in (0, 2, 3))
    return [np.abs(B[k] @ R[k]) for k in (0, 1)], [np.abs(A5[k] @ R[k]) for k in (0, 1)]


@pytest.mark.parametrize("Ls", [5, 8, 16, 20])
def test_every_half_block(Ls):
    """Sites, slices and chiralities of very different size.

    Every half block (12 reals of one site, slice and chirality) is off by at most 1e-14 of the sum of the absolute
    terms that enter it, each taken at the largest entry of its own half block: FP64 rounds about 60 times,
    60 2^-53 = 7e-15; the fixed-point form truncates each half block at 2^-54 and each of Ls products at 2^-57 of
    the largest, less than (4 + Ls) 2^-53 together.
    """
    dims, par = (4, 4, 2, 4), (1.8, 0.03, 1.5, 0.5, "neff", 0.6)
    op, _ = make_pair(dims, Ls, *par, seed=3)
    rng = np.random.default_rng(1)
    x = inputs.gaussian_5d(dims, Ls, 7)
    x *= 2.0 ** rng.integers(-60, 60, x.shape[:5] + (1, 1))
    x[..., 2:, :] *= 2.0 ** rng.integers(-70, 70, x.shape[:5] + (1, 1))
    x[:, 0, ::2] = 0
    fx, ref = both(op, lambda: op.apply(to_gpu(x), op="full", prec="f64"))
    P, A = matrices(dims, Ls, *par)
    X = halves(x)
    mixed = lambda M: np.stack([np.tensordot(M[k], X[k], 1) for k in (0, 1)])
    W = mixed(P).sum(0)   # a neighbour's two chiralities meet in its half spinor
    hop = sum(np.roll(W, d, 1 + ax) for ax in AXIS for d in (1, -1))
    # a row of a unitary link: sum |re| + |im| <= sqrt 6
    bound = mixed(A) + 0.5 * np.sqrt(6.0) * hop
    assert (halves(fx - ref) <= 1e-14 * bound).all()


@pytest.mark.parametrize("k", [-30, -60, -200])
@pytest.mark.parametrize("which", ["P_+", "P_-"])
@pytest.mark.parametrize("dag", [False, True])
def test_small_chirality_beside_a_large_one(k, which, dag):
    """One site and slice, one chirality 2^k below the other: the slice that only the small one reaches through the
    site's own matrix keeps FP64's accuracy (12 products and a sum of 2: 1e-14)."""
    dims, Ls, s = (4, 4, 4, 4), 8, 3
    op, _ = make_pair(dims, Ls, 1.8, 0.03, 1.5, 0.5, "standard", 1.0, seed=3)
    x = np.zeros((Ls,) + dims[::-1] + (4, 3), dtype=np.complex128)
    g = inputs.gaussian_4d((2, 2, 2, 2), 5)[0, 0, 0, 0]
    small, large = (slice(0, 2), slice(2, 4)) if which == "P_+" else (slice(2, 4), slice(0, 2))
    x[s, 1, 2, 3, 0] = g
    x[s, 1, 2, 3, 0, small] *= 2.0 ** k
    fx, ref = both(op, lambda: op.apply(to_gpu(x), op="full", prec="f64", dag=dag))
    for t in (s - 1, s + 1):
        a, b = fx[t, 1, 2, 3, 0, small], ref[t, 1, 2, 3, 0, small]
        assert np.abs(a - b).max() <= 1e-14 * np.abs(b).max(), t
        a, b = fx[t, 1, 2, 3, 0, large], ref[t, 1, 2, 3, 0, large]
        assert np.abs(a - b).max() <= 1e-14 * np.abs(b).max(), t
    assert any(np.abs(ref[t, 1, 2, 3, 0, small]).max() > 0 for t in (s - 1, s + 1))


# ------------------------------------------------------------ extended precision
class Extended:
    """The operator in numpy's extended precision (64 or more bits of mantissa)."""

    def __init__(self, dims, U, Ls, M0, mf, b, c, form, alpha):
        F, C = np.longdouble, np.clongdouble
        self.U = U.astype(C)
        self.U[3, -1] *= -1
        one, K = np.eye(Ls, dtype=F), [np.zeros((Ls, Ls), dtype=F) for _ in range(2)]
        for s in range(Ls):
            K[0][s, s - 1] += F(1) if s else -F(mf)
            K[1][s, (s + 1) % Ls] += F(1) if s < Ls - 1 else -F(mf)
        self.m, self.c = F(4) - F(M0), F(c)
        self.B, self.A = [], []
        for chi in range(2):
            R = one.copy()
            if form == "neff":
                R *= F(alpha)
                w = Ls - 1 if chi == 0 else 0
                R[w, w] = 1
            self.B.append((F(b) * one + F(c) * K[chi]) @ R)
            self.A.append((one - K[chi]) @ R)
        self.inv = [self.inverse(self.m * B + A) for B, A in zip(self.B, self.A)]
        par = np.indices(dims[::-1]).sum(0) % 2
        self.even, self.odd, self.flat = (par == 0)[..., None, None], (par == 1)[..., None, None], par.ravel() == 0
        self.e = [np.array(a, dtype=C) for a in ([[0, -1j], [-1j, 0]], [[0, -1], [1, 0]], [[-1j, 0], [0, 1j]], [[1, 0], [0, 1]])]

    @staticmethod
    def inverse(m):
        n = len(m)
        a = np.concatenate([m, np.eye(n, dtype=m.dtype)], 1)
        for i in range(n):
            p = i + int(np.argmax(abs(a[i:, i])))
            a[[i, p]] = a[[p, i]]
            a[i] /= a[i, i]
            for r in range(n):
                if r != i:
                    a[r] -= a[r, i] * a[i]
        return a[:, n:]

    def hop(self, v):
        out = np.zeros_like(v)
        for mu in range(4):
            g = np.concatenate([np.einsum("ij,...jc->...ic", self.e[mu], v[..., 2:, :]),
                                np.einsum("ij,...jc->...ic", self.e[mu].conj().T, v[..., :2, :])], -2)
            out += np.einsum("...ab,s...ib->s...ia", self.U[mu], np.roll(v - g, -1, 1 + AXIS[mu]))
            out += np.roll(np.einsum("...ba,s...ib->s...ia", self.U[mu].conj(), v + g), 1, 1 + AXIS[mu])
        return out

    @staticmethod
    def fifth(M, v):
        return np.concatenate([np.tensordot(M[0], v[..., :2, :], 1), np.tensordot(M[1], v[..., 2:, :], 1)], -2)

    def full(self, v):
        w = self.fifth(self.B, v)
        return self.m * w - self.hop(w) / 2 + self.fifth(self.A, v)

    def eo(self, v):
        t = self.fifth(self.B, self.fifth(self.inv, self.hop(self.fifth(self.B, v)) * self.odd))
        return v - self.fifth(self.inv, self.hop(t) * self.even) / 4

    def source(self, b4, Ls):
        b5 = np.zeros((Ls,) + b4.shape, dtype=np.clongdouble)
        b5[0, ..., :2, :] = b4[..., :2, :]
        b5[-1, ..., 2:, :] = b4[..., 2:, :]
        return (1 - self.c * self.m) * b5 + self.c / 2 * self.hop(b5)

    def half(self, v):
        return v.reshape(v.shape[0], -1, 4, 3)[:, self.flat]


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 63, reason="no extended precision in numpy here")
@pytest.mark.parametrize("dims,Ls,b,c,form", [((4, 4, 4, 4), 8, 1.0, 0.0, "standard"), ((4, 4, 2, 6), 16, 1.5, 0.5, "neff"),
                                              ((4, 4, 4, 4), 12, 1.0, 1.0, "standard"), ((6, 4, 4, 4), 10, 1.5, 0.5, "neff")])
def test_error_not_above_fp64(dims, Ls, b, c, form):
    """The default's error is not above that of the FP64 kernels: in the norm (whole matrix, even-odd matrix, source),
    and on these fields entry by entry (median, 90 % and 99 % of the reals' relative errors; the source holds zeros)."""
    par = (1.8, 0.02, b, c, form, 0.5)
    U = inputs.random_links(dims, 0.3, 11)
    op, _ = make_pair(dims, Ls, *par, U=U)
    D = Extended(dims, U, Ls, *par)
    x, b4 = inputs.gaussian_5d(dims, Ls, 12), inputs.gaussian_4d(dims, 13)
    xe = D.half(x)
    cases = {"full": (lambda: op.apply(to_gpu(x), op="full", prec="f64"), D.full(x.astype(np.clongdouble))),
             "eo": (lambda: op.apply(to_gpu(xe), op="eo", prec="f64"), D.half(D.eo(x.astype(np.clongdouble) * D.even))),
             "source": (lambda: op.source_5d(to_gpu(b4)), D.source(b4.astype(np.clongdouble), Ls))}
    for name, (call, want) in cases.items():
        err, entries = [], []
        for got in both(op, call):
            d = got.astype(np.clongdouble) - want
            if name != "source":
                r = np.concatenate([abs(d.real / want.real).ravel(), abs(d.imag / want.imag).ravel()]).astype(float)
                entries.append(np.quantile(r, (0.5, 0.9, 0.99)))
            err.append(float(np.sqrt((abs(d) ** 2).sum() / (abs(want) ** 2).sum())))
        print(name, dims, Ls, "default %.3g, FP64 %.3g" % tuple(err))
        assert err[0] <= err[1], name
        assert not entries or (entries[0] <= entries[1]).all(), (name, entries)
