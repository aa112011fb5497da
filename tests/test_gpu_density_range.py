"""GPU tests of the double-float sums far from unit densities: a sum is linear in the density, so its value over a
density scaled by s is s times that over the density itself, to the double-float parity bound (1e-11), as long as products
stay within the float32 exponent range; a mixed solve's velocities scale with the forces to its tolerance."""
import numpy as np
import pytest

import suspensions
from test_gpu_corrections import bodies, lattice, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rbs():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1606_07428_gb300 import rbs as m
    return m


def chains(p=6):
    c = lattice((5, 1, 1), 2.4)
    return bodies(np.concatenate([c, c + [60.0, 0, 0]]), p, (1.0, 0.9, 0.8), True)


@pytest.mark.parametrize("far", ["DIRECT", "TREECODE_DF"])
@pytest.mark.parametrize("scale", [1e-26, 1e-22, 1e-20, 1e19, 1e20, 1e22, 1e26])
def test_operators_scale_with_the_density(rbs, far, scale):
    s = chains()
    x = suspensions.random_density(21, s.total_nodes)
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED, far_field=getattr(rbs, f"RBS_FAR_{far}"), tree_df_theta=0.6,
                     tree_df_degree=5) as ctx:
        ctx.set_suspension(s)
        st = rbs.rbs_get_stats(ctx.ctx)
        assert st["near_pairs"] > 0 and (far == "DIRECT" or st["tree_df_proxy_pairs"] > 0)
        for op in (rbs.RBS_OP_K_OFF, rbs.RBS_OP_S_OFF):
            y = rbs.rbs_apply_operator(ctx.ctx, op, rbs.RBS_PREC_DF, x)
            assert rel(rbs.rbs_apply_operator(ctx.ctx, op, rbs.RBS_PREC_DF, scale * x) / scale, y) < 1e-11


@pytest.mark.parametrize("scale", [1e-22, 1e22])
def test_solves_scale_with_the_forces(rbs, scale):
    s = chains()
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED) as ctx:
        ctx.set_suspension(s)
        v, om, _, _ = rbs.rbs_mobility_solve(ctx.ctx, s.F, s.T, 1e-10)
        vs, oms, _, _ = rbs.rbs_mobility_solve(ctx.ctx, scale * s.F, scale * s.T, 1e-10)
        assert rel(np.concatenate([vs, oms]) / scale, np.concatenate([v, om])) < 1e-9
