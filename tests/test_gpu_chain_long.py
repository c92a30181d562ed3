"""Chains that do not fit one launch, or one window of subgraphs, against the FP64 oracle.

A launch holds 96 products and a window about three tiles an SM, in both forms.  Bounds: in a gap at a few K the worst
case of FP32 sums, every product of the recursion off by n 2^-24 (about 100 products of n = 132: 8e-4 e; a product left
out, repeated or begun too early is off by the size of a charge); at 300 K the 2e-5 e of forms 1 and 4.
"""
import numpy as np
import pytest

from oracle import density as odn
from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,Te", [(1, 4.6875), (4, 18.75)])       # 16 and 14 doublings
def test_more_products_than_a_launch_holds(precision, Te):
    from paper_2606_03140_gb300 import sedacs as S

    s = I.small_water_box(22, (29.97 * 22) ** (1 / 3), 722)
    n = I.random_charges(s.n_atoms, 5, 0.02)
    cores, halos = odn.full_partition(s.n_atoms)
    m = I.default_model()
    warm = odn.density(s.R, s.species, s.box, m, n, cores, halos)
    e = warm.subs[0].eps
    top, bot = np.max(e[e < warm.mu]), np.min(e[e > warm.mu])
    assert bot - top > 0.1
    mu = 0.5 * (top + bot)
    ref = odn.density(s.R, s.species, s.box, m, n, cores, halos, Te=Te, mu=mu)
    ctx = S.sedacs_create(s.species, s.box, m, S.sedacs_default_params(precision=precision, Te=Te, mu_given=1))
    try:
        R = np.ascontiguousarray(s.R)
        S.sedacs_graph_build(ctx, R)
        S.sedacs_set_cores(ctx, cores)
        _, q, _, _ = S.sedacs_subgraph_density(ctx, R, n, mu)
        doublings = S.sedacs_density_info(ctx)["doublings"]
    finally:
        S.sedacs_destroy(ctx)
    products = 6 + (6 if precision == 1 else 7) * doublings - 1       # of the recursion, but the last one
    assert products > 96
    assert np.max(np.abs(q - ref.q)) < products * 132 * 2.0**-24


@pytest.mark.parametrize("precision", [1, 4])
def test_more_subgraphs_than_a_window_holds(precision):
    from paper_2606_03140_gb300 import sedacs as S

    s = I.small_water_box(64, (29.97 * 64) ** (1 / 3), 764)
    n = I.random_charges(s.n_atoms, 5, 0.02)
    # every pair of atoms is an edge, so each of the 128 subgraphs is the whole box (384 orbitals, six tiles)
    cut = np.cumsum([0] + [1, 2] * 64)
    cores = [np.arange(a, b, dtype=np.int32) for a, b in zip(cut[:-1], cut[1:])]
    ref = odn.density(s.R, s.species, s.box, I.default_model(), n, *odn.full_partition(s.n_atoms))
    ctx = S.sedacs_create(s.species, s.box, I.default_model(), S.sedacs_default_params(precision=precision, r_graph=30.0))
    try:
        R = np.ascontiguousarray(s.R)
        assert S.sedacs_graph_build(ctx, R) == s.n_atoms * (s.n_atoms - 1)
        S.sedacs_set_cores(ctx, cores)
        _, q, _, _ = S.sedacs_subgraph_density(ctx, R, n)
    finally:
        S.sedacs_destroy(ctx)
    assert np.max(np.abs(q - ref.q)) < 2e-5
