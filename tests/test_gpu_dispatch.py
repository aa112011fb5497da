"""GPU tests of the direct float32 sums' size rule: small systems take one target per lane, larger ones two
(rbs_stats.pair_variant 9 and 10), by themselves and where rbs_options.pair_variant asks; either form is within the
float32 operator bound (2e-5) of the float64 operators."""
import pytest

import suspensions
from test_gpu_corrections import rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rbs():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1606_07428_gb300 import rbs as m
    return m


@pytest.mark.parametrize("n,p,option,form", [(2, 4, 0, 9), (8, 8, 0, 9), (101, 8, 0, 10), (40, 10, 0, 10), (8, 8, 2, 10),
                                             (101, 8, 1, 9)])
def test_direct_float32_sums_by_size(rbs, n, p, option, form):
    s = suspensions.random_ellipsoids(n, p, 2 * p, 0.10, 0.2, seed=31)
    x = suspensions.random_density(32, s.total_nodes)
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED, pair_variant=option) as ctx:
        ctx.set_suspension(s)
        assert rbs.rbs_get_stats(ctx.ctx)["pair_variant"][:2] == [form, form]
        for op in (rbs.RBS_OP_K_OFF, rbs.RBS_OP_S_OFF):
            y = rbs.rbs_apply_operator(ctx.ctx, op, rbs.RBS_PREC_MIXED, x)
            assert rel(y, rbs.rbs_apply_operator(ctx.ctx, op, rbs.RBS_PREC_FP64, x)) < 2e-5
