"""GPU tests of the double-float sums that leave out the sources near a target's particle.

* Against the float64 operators where the lists are at their edges: particles of 12 and 24 nodes (four and two of them
  in a unit of targets), more than 32 near sources per target, every particle near every other, none near, suspensions
  of one context.  A separation is rounded to 2^-48 of coordinates of up to four radii, its fifth power makes that
  2^-48 * 20 / gap of a term, and three such roundings (the pair's, the powers' and the sums') stay within
  2^-48 * 64 / gap; the gaps here are 0.5 or more.
* The scalar operators over the same lists, against the oracle's dense ones (1e-11, the magnetostatic parity bound).
"""
import numpy as np
import pytest

import oracle
import suspensions
from oracle import magnetic as om
from test_gpu_corrections import bodies, lattice, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rbs():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1606_07428_gb300 import rbs as m
    return m


def compare(rbs, ctx, x, tol):
    for op in (rbs.RBS_OP_K_OFF, rbs.RBS_OP_S_OFF):
        y = rbs.rbs_apply_operator(ctx.ctx, op, rbs.RBS_PREC_DF, x)
        assert rel(y, rbs.rbs_apply_operator(ctx.ctx, op, rbs.RBS_PREC_FP64, x)) < tol


@pytest.mark.parametrize("near_delta", [0.0, 1.0, 2.5, 20.0])
@pytest.mark.parametrize("shape,p,nphi", [((5, 5, 4), 2, 4), ((4, 4, 4), 3, 6), ((4, 3, 3), 5, 14), ((3, 3, 2), 8, 16)])
def test_double_float_sums_at_the_edges_of_the_near_lists(rbs, shape, p, nphi, near_delta):
    c = lattice(shape, 2.9)
    s = bodies(c[np.random.default_rng(2).permutation(len(c))], p, (1.2, 0.8, 0.9), True)
    n = s.n
    ids = np.repeat([0, 1, 2], [1, 5, n - 6]).astype(np.int32)
    for sid in (None, ids):
        with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED, near_delta=near_delta) as ctx:
            ctx.set_geometry(s.semi_axes, s.p, np.full(n, nphi, np.int32), s.centres, s.quats, sid)
            compare(rbs, ctx, suspensions.random_density(18, n * (p + 1) * nphi), 2.0 ** -48 * 64 / 0.5)


@pytest.mark.parametrize("shape,p,delta", [((3, 3, 5), 2, 9.0), ((3, 3, 2), 3, 1.0), ((2, 2, 2), 5, 0.0)])
def test_scalar_sums_leave_near_sources_out(rbs, shape, p, delta):
    s = bodies(lattice(shape, 2.9), p, (1.2, 0.8, 0.9), True)
    dense = om.Magnetic(oracle.System(s.semi_axes, s.p, s.nphi, s.centres, s.quats, options=oracle.Options(delta=delta)))
    x = np.random.default_rng(3).normal(size=s.total_nodes)
    with rbs.Context(device=0, near_delta=delta) as ctx:
        ctx.set_suspension(s)
        for kind in (0, 1):
            assert rel(rbs.rbs_apply_laplace(ctx.ctx, kind, x), dense.assemble("KS"[kind]) @ x) < 1e-11
