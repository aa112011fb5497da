"""GPU tests of the refinement's cheap updates: r -= A d and u += S d with float32 sums between particles that
are not near (the mixed solve's later refinements).

A solve's tolerance is on ||b - A mu|| / ||b||, and the updates may cost a tenth of it, at every gap: the float64
residual of the density returned stays within 1.1 tol, as does the reported one's distance from it.  Passes and
updates are counted (each refinement is one or the other), so that a solve without updates fails.
"""
import numpy as np
import pytest

import suspensions

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def rbs():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1606_07428_gb300 import rbs as m
    return m


def rel(a, b):
    return np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b))


def lattice(shape, spacing):
    return np.stack(np.meshgrid(*[np.arange(k) * spacing for k in shape], indexing="ij"), -1).reshape(-1, 3)


def bodies(centres, p, axes=(1.0, 1.0, 1.0), turned=False, seed=0):
    n, rng = len(centres), np.random.default_rng(seed)
    quats = suspensions.random_quaternions(rng, n) if turned else np.tile([1.0, 0, 0, 0], (n, 1))
    return suspensions.Suspension(np.tile(axes, (n, 1)), np.full(n, p, np.int32), np.full(n, 2 * p, np.int32),
                                  np.asarray(centres, float), quats, rng.normal(size=(n, 3)), rng.normal(size=(n, 3)),
                                  np.zeros(n, np.int32))


def geometry(name, gap):
    if name == "row":          # equal orientation: nodes face one another across every gap
        return bodies(lattice((4, 1, 1), 2 + gap), 8)
    if name == "one pair":     # one close pair among spread spheres, last in the order
        return bodies(np.concatenate([lattice((4, 2, 2), 3.2), [[-4.0, 0, 0], [-6.0 - gap, 0, 0]]]), 6)
    if name == "shuffled":     # neighbours far apart in the particle order, units of targets across particles
        return bodies(lattice((4, 3, 3), 2.6 + gap)[np.random.default_rng(1).permutation(36)], 5, (1.3, 0.8, 1.0), True)
    return bodies(lattice((2, 2, 2), 2 + gap), 6, (1.0, 0.7, 0.8), True)  # turned


def solve(rbs, ctx, s):
    rbs.rbs_reset_stats(ctx.ctx)
    v, om, mu, _ = rbs.rbs_mobility_solve(ctx.ctx, s.F, s.T, TOL, want_density=True)
    st = rbs.rbs_get_stats(ctx.ctx)
    passes = st["kernel_count"][rbs.RBS_KC_PAIR_KSDF]
    assert st["kernel_count"][rbs.RBS_KC_PAIR_S32] == 0  # no Stokeslet sum of the float32 operator enters u
    return v, om, mu, st["residual"], passes, st["refinements"] - passes


def check_residual(rbs, ctx, s, out, prec):
    """The residual of the solve's density by the operators of ctx in prec; returns the incident density."""
    mu, reported = out[2], out[3]
    rho = rbs.rbs_incident_density(ctx.ctx, s.F, s.T)
    b = -rbs.rbs_apply_operator(ctx.ctx, rbs.RBS_OP_HALF_K, prec, rho)
    r = b - rbs.rbs_apply_operator(ctx.ctx, rbs.RBS_OP_A, prec, mu)
    true = np.linalg.norm(r) / np.linalg.norm(b)
    assert true <= 1.1 * TOL and abs(true - reported) <= 0.11 * TOL
    return rho


def check(rbs, ctx, s, out, prec):
    """The same, and the velocities of that density."""
    v, om, mu = out[:3]
    u = rbs.rbs_apply_operator(ctx.ctx, rbs.RBS_OP_S, prec, check_residual(rbs, ctx, s, out, prec) + mu)
    assert rel(np.concatenate([v, om]), np.concatenate(rbs.rbs_rigid_velocities(ctx.ctx, u, s.n))) < 0.1 * TOL


@pytest.mark.parametrize("name", ["row", "one pair", "shuffled", "turned"])
@pytest.mark.parametrize("gap", [0.2, 0.1, 0.05, 0.02, 0.01])
@pytest.mark.parametrize("far", ["DIRECT", "TREECODE_DF"])
def test_updates_keep_the_tolerance_at_every_gap(rbs, name, gap, far):
    s = geometry(name, gap)
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED, far_field=getattr(rbs, f"RBS_FAR_{far}")) as ctx, \
            rbs.Context(device=0) as exact:
        ctx.set_suspension(s)
        exact.set_suspension(s)
        out = solve(rbs, ctx, s)
        assert out[4] >= 1 and out[5] >= 1
        check(rbs, exact, s, out, rbs.RBS_PREC_FP64)


@pytest.mark.parametrize("far", ["DIRECT", "TREECODE_DF"])
def test_passes_keep_the_tolerance_at_a_tiny_gap(rbs, far):
    # what a double-float pass adds for a near pair and removes again would be 1e-9 of the residual here
    s = geometry("one pair", 0.003)
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED, far_field=getattr(rbs, f"RBS_FAR_{far}")) as ctx, \
            rbs.Context(device=0) as exact:
        ctx.set_suspension(s)
        exact.set_suspension(s)
        check_residual(rbs, exact, s, solve(rbs, ctx, s), rbs.RBS_PREC_FP64)


@pytest.mark.parametrize("degree", [2, 3, 5, 8, 12])
def test_updates_over_clusters(rbs, degree):
    # close pairs in two chains that see one another as clusters; the same lists in double-float are the reference
    m = 17 if degree > 8 else 14  # more nodes in a chain than proxy points, so that it is one cluster
    x = np.concatenate([np.arange(m) * 2.05, np.arange(m) * 2.05 + 5.0 * m])
    s = bodies(np.stack([x, 0 * x, 0 * x], 1), 8 if degree > 8 else 6, seed=3)
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED, far_field=rbs.RBS_FAR_TREECODE_DF, tree_df_theta=0.6,
                     tree_df_degree=degree) as ctx:
        ctx.set_suspension(s)
        assert rbs.rbs_get_stats(ctx.ctx)["tree_df_proxy_pairs"] > 0
        out = solve(rbs, ctx, s)
        assert out[4] >= 1 and out[5] >= 1
        check(rbs, ctx, s, out, rbs.RBS_PREC_DF)


@pytest.mark.parametrize("degree", [4, 7, 8, 10])
@pytest.mark.parametrize("gap", [0.2, 0.02])
def test_small_updates_over_the_float32_treecode(rbs, degree, gap):
    # 16-bit blocks: several refinements, the last ones small enough for the float32 lists; passes are direct
    m = 18  # particles of 84 nodes: more nodes in a chain than the 1,331 proxy points of degree 10
    x = np.concatenate([np.arange(m) * (2 + gap), np.arange(m) * (2 + gap) + 6.0 * m])
    s = bodies(np.stack([x, 0 * x, 0 * x], 1), 6, seed=4)
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED_BF16, far_field=rbs.RBS_FAR_TREECODE, tree_theta=0.6,
                     tree_degree=degree) as ctx, rbs.Context(device=0) as exact:
        ctx.set_suspension(s)
        exact.set_suspension(s)
        assert rbs.rbs_get_stats(ctx.ctx)["tree_proxy_pairs"] > 0
        out = solve(rbs, ctx, s)
        assert out[4] >= 1 and out[5] >= 1
        check(rbs, exact, s, out, rbs.RBS_PREC_FP64)


def test_no_update_without_a_near_margin(rbs):
    # near_delta 0: particles that are not near may be as close as they like
    s = geometry("turned", 0.3)
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED, near_delta=0.0) as ctx, \
            rbs.Context(device=0, near_delta=0.0) as exact:
        ctx.set_suspension(s)
        exact.set_suspension(s)
        out = solve(rbs, ctx, s)
        assert out[5] == 0
        check(rbs, exact, s, out, rbs.RBS_PREC_FP64)
