"""The P2 velocity kernels one by one: a stencil sweep against a numpy product
of the exported blocks and, bit for bit, against the 2x2-block SELL sweep
(the same sums in the same order) on every level, in its four epilogues and
three starts, FP32 and BF16 values, both top conditions and a non-square box,
at sizes that reach one cell a thread (256) and 2, 4 and 8 warps a row (176,
128, 6); the grid transfers against the oracle's; the dense inverse of a
coarsest level by a cluster and by one block."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import mg
from oracle.mesh import Mesh
from paper_2501_11767_gb300 import chnss, inputs

pytestmark = pytest.mark.gpu

EPS = {0: 2.0 ** -53, 1: 2.0 ** -24}
COEF = [0.37, 1.21, -0.43, 0.77]                    # scale, c0, c1, c2


def _context(n, top_bc, lxy):
    p = inputs.default_params()
    p.update(top_bc=top_bc)
    ctx = chnss.Context(chnss.Mesh(n, *lxy, top_bc=top_bc), p)
    st = inputs.initial_state(n, seed=3)
    st["v"] = 0.02 * np.random.default_rng(n).standard_normal(2 * ctx.mesh.N2)
    ctx.assemble(chnss.state_to_device(st))
    return ctx


def _rounded(a, precision):
    """FP64 values in FP32, or to the eight significand bits of BF16 (to nearest even)."""
    if precision == 1:
        return a.astype(np.float32).astype(np.float64)
    m, e = np.frexp(a)
    return np.ldexp(np.rint(m * 256) / 256, e)


def _vectors(size, seed):
    rng = np.random.default_rng(seed)
    v = [rng.standard_normal(size).astype(np.float32).astype(np.float64) for _ in range(4)]
    return v[0], v[1], v[2], np.abs(v[3]) + 0.5     # u, b, w, dinv


FORMS = [(0, 0, False), (1, 0, False), (2, 0, False), (3, 0, False), (3, 0, True), (3, 1, False), (3, 2, False)]


@pytest.mark.parametrize("n,lxy,warps", [(2, (1.0, 1.0), 8), (6, (1.0, 1.0), 8), (10, (2.0, 0.75), 8),
                                         (128, (1.0, 1.0), 4), (176, (0.3, 0.7), 2), (256, (1.0, 1.0), 1)])
@pytest.mark.parametrize("top_bc", [0, 1])
def test_sweep(n, lxy, warps, top_bc):
    ctx = _context(n, top_bc, lxy)
    rp, col, val = ctx.export_csr(chnss.MAT_A)
    eps = EPS[1]
    c = np.asarray(COEF, dtype=np.float32).astype(np.float64)
    for level in range(ctx.mesh.levels):
        size = 2 * (2 * (n >> level) + 1) ** 2
        u, b, w, d = _vectors(size, 10 * n + level)
        # the first iterate by the sweep's two multiplications
        x1 = ((np.float32(c[0]) * d.astype(np.float32)) * b.astype(np.float32)).astype(np.float64)
        for precision in (1, 2):
            if level == 0:
                A = sp.csr_matrix((_rounded(val, precision), col, rp), shape=(size, size))
                absA = abs(A)
            for mode, start, with_w in FORMS:
                args = dict(b=b, dinv=d, coef=COEF)
                uu = x1 if start == 1 else u
                ww = x1 if start == 2 else w if with_w else None
                got, k = ctx.debug_velocity_sweep(level, 1, precision, mode, u, w=w if with_w else None, out=w,
                                                  start=start, **args)
                same, _ = ctx.debug_velocity_sweep(level, 0, precision, mode, uu, w=ww, out=w, **args)
                where = (level, precision, mode, start, with_w)
                assert np.isfinite(got).all() and np.array_equal(got, same), where
                if level:
                    continue
                assert k == warps
                au, mag = A @ uu, absA @ np.abs(uu)
                if mode == 0:
                    want, scale = au, mag
                elif mode == 1:
                    want, scale = b - au, mag + np.abs(b)
                elif mode == 2:
                    want, scale = w + au, mag + np.abs(w)
                else:
                    want = c[1] * uu + c[3] * d * (b - au)
                    scale = np.abs(c[1] * uu) + np.abs(c[3] * d) * (np.abs(b) + mag)
                    if ww is not None:
                        want, scale = want + c[2] * ww, scale + np.abs(c[2] * ww)
                # sums of at most 38 products and six more roundings
                assert (np.abs(got - want) <= 48 * eps * scale).all(), where


@pytest.mark.parametrize("top_bc", [0, 1])
@pytest.mark.parametrize("n", [4, 6, 10, 44, 200])         # 200: lines of more than one block of threads
def test_transfers(n, top_bc):
    ctx = _context(n, top_bc, (1.0, 1.0))
    fine, coarse = (Mesh(k, top_free=top_bc == 1) for k in (n, n // 2))
    P = mg.prolongation_velocity(coarse, fine)
    rng = np.random.default_rng(n)
    for precision in (0, 1):
        t = np.float32 if precision else np.float64
        r, x = (rng.standard_normal(k).astype(t).astype(np.float64) for k in P.shape)
        got = ctx.debug_velocity_transfer(0, precision, False, r)
        want = P.T @ r
        # at most 25 terms with exact weights
        assert (np.abs(got - want) <= 26 * EPS[precision] * (abs(P.T) @ np.abs(r))).all(), precision
        got = ctx.debug_velocity_transfer(0, precision, True, x, out=r)
        want = r + P @ x
        assert (np.abs(got - want) <= 8 * EPS[precision] * (np.abs(r) + abs(P) @ np.abs(x))).all(), precision


@pytest.mark.parametrize("n", [1, 2, 50, 97, 98, 127, 128, 129, 224, 225, 242, 256])
def test_dense_inverse(n):
    """Off-diagonal entries dominate, so rows are exchanged; with unit pairs
    the remaining rows have to give the same bits as without the mask."""
    rng = np.random.default_rng(n)
    base = rng.uniform(-1, 1, (n, n))
    base[np.arange(n), np.arange(n)] *= 1e-3
    masks = [None]
    if n % 2 == 0:
        pairs = n // 2
        masks += [np.arange(pairs) < max(pairs // 3, 1), np.arange(pairs) >= pairs - max(pairs // 3, 1),
                  np.ones(pairs, bool), np.arange(pairs) % 3 == 1, np.arange(pairs) % 2 == 0]
    for mask in masks:
        A = base.copy()
        if mask is not None:
            at = np.flatnonzero(np.repeat(mask, 2))
            A[at] = 0.0
            A[:, at] = 0.0
            A[at, at] = 1.0
        ref = np.linalg.inv(A)
        one, st1 = chnss.debug_dense_inverse(A, False)
        got, st = chnss.debug_dense_inverse(A, True)
        assert st == 0 and st1 == 0
        # backward error of elimination with row exchanges, growth below 2 n on such matrices
        tol = 4 * n * n * np.finfo(float).eps * np.linalg.cond(A)
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
        assert np.array_equal(got, one)
        if mask is not None:
            skipped, st = chnss.debug_dense_inverse(A, True, unit=mask)
            assert st == 0 and np.array_equal(skipped, got)


def test_zero_pivot_is_reported():
    A = np.eye(40) + np.eye(40, k=1)
    A[:, 17] = 0.0
    assert chnss.debug_dense_inverse(A, True)[1] == 1
    assert chnss.debug_dense_inverse(A, False)[1] == 1
