"""One V-cycle with thread-block clusters and without them (the forms that run
where the device has no place for a cluster): the same bits, since every row
is summed and stepped by the same expressions in the same order, for the P1
and velocity hierarchies, FP64, FP32 and BF16 values, both top conditions,
one to three vectors, and the query that decides."""
import numpy as np
import pytest

from paper_2501_11767_gb300 import chnss, inputs

pytestmark = pytest.mark.gpu


def _context(n, top_bc, precision=0, lxy=(1.0, 1.0)):
    p = inputs.default_params()
    p.update(top_bc=top_bc, precision=precision)
    ctx = chnss.Context(chnss.Mesh(n, *lxy, top_bc=top_bc), p)
    st = inputs.initial_state(n, seed=2)
    st["v"] = 0.02 * np.random.default_rng(n).standard_normal(2 * ctx.mesh.N2)
    ctx.assemble(chnss.state_to_device(st))
    return ctx


def _random(n, seed):
    return np.random.default_rng(seed).standard_normal(n)


# levels taken, by the sizes: the largest of at most 128 (FP32) or 64 (FP64) cells a side
@pytest.mark.parametrize("top_bc", [0, 1])
@pytest.mark.parametrize("n", [4, 10, 18, 34, 44, 50, 64, 88, 104, 128, 136, 200, 256])
def test_p1_cycles(n, top_bc):
    ctx = _context(n, top_bc)
    for block in (0, 2):
        for precision, largest in ((0, 64), (1, 128)):
            b = _random(3 * ctx.mesh.N1, n)
            one = b[:ctx.mesh.N1]
            got, first, tail, inv, _ = ctx.debug_vcycle(block, precision, True, one)
            want, none, _, noinv, _ = ctx.debug_vcycle(block, precision, False, one)
            cells = [n >> l for l in range(20) if n >> l << l == n]
            cells = cells[:next((i for i, c in enumerate(cells) if c % 2 or c <= 2), len(cells) - 1) + 1]
            assert first == next((i for i, c in enumerate(cells[:-1]) if c <= largest), -1), cells
            assert none == -1 and noinv in (0, -1) and inv in (0, 1, -1)
            assert np.isfinite(got).all() and np.array_equal(got, want), (block, precision)
            if block == 0:
                for nvec in (1, 2, 3):
                    many, mfirst, *_ = ctx.debug_vcycle(0, precision, True, b[:nvec * ctx.mesh.N1], nvec)
                    plain, mnone, *_ = ctx.debug_vcycle(0, precision, False, b[:nvec * ctx.mesh.N1], nvec)
                    assert (mfirst == -1) == (first == -1) and mnone == -1
                    assert np.array_equal(many, plain), (precision, nvec)
                    assert np.array_equal(many[:ctx.mesh.N1], got), (precision, nvec)


@pytest.mark.parametrize("lxy", [(1.0, 1.0), (0.3, 0.7)])
@pytest.mark.parametrize("top_bc", [0, 1])
@pytest.mark.parametrize("n", [4, 8, 14, 16, 20, 22, 24, 32, 34, 48, 50, 80, 128])
def test_velocity_cycles(n, top_bc, lxy):
    ctx = _context(n, top_bc, lxy=lxy)
    b = _random(2 * ctx.mesh.N2, n)
    for precision in (1, 2):
        got, first, _, inv, stencils = ctx.debug_vcycle(1, precision, True, b)
        want, none, _, noinv, same = ctx.debug_vcycle(1, precision, False, b)
        assert first >= 0 and none == -1 and noinv in (0, -1)
        assert stencils == same and stencils > first
        assert np.isfinite(got).all() and np.array_equal(got, want), precision


def test_velocity_fp64_inverse():
    """The FP64 hierarchy has no velocity cluster; its dense inverse is one's."""
    ctx = _context(20, 0)
    b = _random(2 * ctx.mesh.N2, 1)
    got, first, _, inv, stencils = ctx.debug_vcycle(1, 0, True, b)
    want, _, _, noinv, _ = ctx.debug_vcycle(1, 0, False, b)
    assert (first, inv, noinv, stencils) == (-1, 1, 0, 0)
    assert np.array_equal(got, want)


def test_query():
    assert chnss.debug_cluster_runs(16, 512, 64 << 10)       # about what the inverse of 240 rows asks for
    assert not chnss.debug_cluster_runs(64, 512, 1 << 10)    # more blocks than a cluster can have
    assert not chnss.debug_cluster_runs(16, 512, 1 << 20)    # more shared memory than a block can have
    with pytest.raises(chnss.ChnssError):
        chnss.debug_cluster_runs(0, 512, 0)
