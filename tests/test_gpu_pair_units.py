"""GPU parity of the pair sums at the edges of their work units and of the proxy grids.

* Treecode clusters at the degrees whose tensor grids differ in form (odd and even point counts, the
  smallest, the default, the largest of each arithmetic), for particles whose node counts leave 8 to 32
  targets in a unit, against the oracle's statement of the same treecode: float32 within 2e-6, double-float
  within 1e-11, the bounds of the treecode parity tests.
* Direct sums over particles of 8 to 60 nodes (one to two units of a particle, sources split over half-warps),
  with and without near pairs: float64 1e-12, double-float 1e-11, float32 2e-5, the operator parity bounds.
* Double-float sums against float64 ones: the separation, its powers and the sums carry 44 bits and more, so the
  relative L2 gap stays below 2^-41 = 4.5e-13 even where near particles meet far ones in a tile.
* The singular rule in two factors for rules of other orders than the default, against the oracle's blocks (1e-12).
* A mixed solve whose last correction is applied by the cheaper operator: the float64 residual of the density
  stays within the tolerance and the tenth of it that the updates may cost.
"""
import numpy as np
import pytest

import oracle
import suspensions
from oracle import treecode as tc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rbs():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1606_07428_gb300 import rbs as m
    return m


def rel(a, b):
    return np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b))


def two_chains(m, p, nphi, seed):
    """Two collinear chains of m ellipsoids, 3.2 apart in a chain, far enough apart for either to be one cluster."""
    rng = np.random.default_rng(seed)
    x = np.concatenate([np.arange(m) * 3.2, np.arange(m) * 3.2 + 8.0 * m + 12.0])
    centres = np.stack([x, 0 * x, 0 * x], 1)
    axes = rng.uniform(0.6, 1.4, size=(2 * m, 3))
    quats = suspensions.random_quaternions(rng, 2 * m)
    F = rng.normal(size=(2 * m, 3))
    return suspensions.Suspension(axes, np.full(2 * m, p, np.int32), np.full(2 * m, nphi, np.int32), centres, quats, F, F,
                                  np.zeros(2 * m, np.int32))


def off_diagonal(ref, kind, x):
    y = np.zeros_like(x)
    for i in range(len(ref.particles)):
        for j in range(len(ref.particles)):
            if j != i:
                y[ref.sl(i)] += np.einsum("tkms,sm->tk", ref.pair_block(kind, i, j), x[ref.sl(j)])
    return y


@pytest.mark.parametrize("arithmetic,degree,m,p,nphi", [
    ("float32", 2, 3, 4, 8), ("float32", 4, 6, 5, 10), ("float32", 6, 8, 6, 12), ("float32", 7, 5, 8, 16),
    ("float32", 8, 8, 8, 16), ("float32", 10, 11, 8, 16), ("double-float", 2, 3, 4, 8), ("double-float", 5, 5, 6, 14),
    ("double-float", 11, 13, 8, 16), ("double-float", 12, 17, 8, 16)])
def test_cluster_sums_match_the_oracle(rbs, arithmetic, degree, m, p, nphi):
    s = two_chains(m, p, nphi, 100 + degree)
    ref = oracle.System(s.semi_axes, s.p, s.nphi, s.centres, s.quats)
    tree = tc.Treecode(ref, 0.6, degree)
    assert tree.pair_counts()[1] > 0
    x = suspensions.random_density(41, s.total_nodes)
    f32 = arithmetic == "float32"
    kw = {"far_field": rbs.RBS_FAR_TREECODE, "tree_theta": 0.6, "tree_degree": degree} if f32 else \
         {"far_field": rbs.RBS_FAR_TREECODE_DF, "tree_df_theta": 0.6, "tree_df_degree": degree}
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED, **kw) as ctx:
        ctx.set_suspension(s)
        st = rbs.rbs_get_stats(ctx.ctx)
        assert st["tree_proxy_pairs" if f32 else "tree_df_proxy_pairs"] == tree.pair_counts()[1]
        for kind in ("K", "S"):
            y = rbs.rbs_apply_operator(ctx.ctx, getattr(rbs, f"RBS_OP_{kind}_OFF"),
                                       rbs.RBS_PREC_MIXED if f32 else rbs.RBS_PREC_DF, x)
            want = tc.offdiagonal_with_tree(ref, tree, kind, x)
            assert rel(y, want) < (2e-6 if f32 else 1e-11)


@pytest.mark.parametrize("gap,fill", [(0.2, 0.12), (2.5, 0.02)])
@pytest.mark.parametrize("p,nphi", [(2, 4), (3, 4), (4, 8), (5, 10)])
def test_direct_sums_at_unit_edges(rbs, p, nphi, gap, fill):
    nphi = max(nphi, 2 * p)
    s = suspensions.random_ellipsoids(5, p, nphi, fill, gap, seed=50 + p)
    ref = oracle.System(s.semi_axes, s.p, s.nphi, s.centres, s.quats)
    x = suspensions.random_density(42, s.total_nodes)
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED) as ctx:
        ctx.set_suspension(s)
        for kind in ("K", "S"):
            want = off_diagonal(ref, kind, x)
            op = getattr(rbs, f"RBS_OP_{kind}_OFF")
            for prec, tol in ((rbs.RBS_PREC_FP64, 1e-12), (rbs.RBS_PREC_DF, 1e-11), (rbs.RBS_PREC_MIXED, 2e-5)):
                assert rel(rbs.rbs_apply_operator(ctx.ctx, op, prec, x), want) < tol


@pytest.mark.parametrize("n,p,seed", [(64, 8, 12), (33, 10, 13), (150, 6, 14)])
def test_double_float_sums_against_float64(rbs, n, p, seed):
    s = suspensions.random_ellipsoids(n, p, 2 * p, 0.10, 0.2, seed=seed)
    x = suspensions.random_density(seed, s.total_nodes)
    with rbs.Context(device=0) as ctx:
        ctx.set_suspension(s)
        for op in (rbs.RBS_OP_K_OFF, rbs.RBS_OP_S_OFF):
            y = rbs.rbs_apply_operator(ctx.ctx, op, rbs.RBS_PREC_DF, x)
            assert rel(y, rbs.rbs_apply_operator(ctx.ctx, op, rbs.RBS_PREC_FP64, x)) < 2.0 ** -41


@pytest.mark.parametrize("p,nphi,factor", [(2, 4, 1), (5, 10, 1), (4, 10, 3), (7, 14, 4)])
def test_singular_rule_of_other_orders(rbs, p, nphi, factor):
    s = suspensions.random_ellipsoids(2, p, nphi, 0.02, 2.5, seed=60 + p)
    ref = oracle.System(s.semi_axes, s.p, s.nphi, s.centres, s.quats, options=oracle.Options(p_self_factor=factor))
    x = suspensions.random_density(43, s.total_nodes)
    with rbs.Context(device=0, p_self_factor=factor) as ctx:
        ctx.set_suspension(s)
        for kind in ("K", "S"):
            y = rbs.rbs_apply_operator(ctx.ctx, getattr(rbs, f"RBS_OP_{kind}_SELF"), rbs.RBS_PREC_FP64, x)
            want = np.concatenate([(ref.self_block_lab(kind, i) @ x[ref.sl(i)].ravel()).reshape(-1, 3) for i in range(2)])
            assert rel(y, want) < 1e-12


@pytest.mark.parametrize("far", ["DIRECT", "TREECODE"])
@pytest.mark.parametrize("seed", [71, 72])
def test_corrected_solve_meets_its_tolerance(rbs, far, seed):
    tol = 1e-10
    s = suspensions.random_ellipsoids(60, 6, 12, 0.12, 0.2, seed=seed)
    with rbs.Context(device=0, precision=rbs.RBS_PREC_MIXED, far_field=getattr(rbs, f"RBS_FAR_{far}"), tree_degree=4) as ctx, \
            rbs.Context(device=0) as exact:
        ctx.set_suspension(s)
        exact.set_suspension(s)
        v, om, mu, _ = rbs.rbs_mobility_solve(ctx.ctx, s.F, s.T, tol, want_density=True)
        rho = rbs.rbs_incident_density(exact.ctx, s.F, s.T)
        b = -rbs.rbs_apply_operator(exact.ctx, rbs.RBS_OP_HALF_K, rbs.RBS_PREC_FP64, rho)
        r = b - rbs.rbs_apply_operator(exact.ctx, rbs.RBS_OP_A, rbs.RBS_PREC_FP64, mu)
        assert np.linalg.norm(r) <= 1.15 * tol * np.linalg.norm(b)
        u = rbs.rbs_apply_operator(exact.ctx, rbs.RBS_OP_S, rbs.RBS_PREC_FP64, rho + mu)
        ve, ome = rbs.rbs_rigid_velocities(exact.ctx, u, s.n)
        # the velocities of the solve are those of its own density, to the updates' share of the tolerance
        assert rel(np.concatenate([v, om]), np.concatenate([ve, ome])) < tol
