"""D_c and W_c after an accepted step of the chemical potential, term by term, against the oracle's levels.

At 30,000 K the levels next to mu are partly filled, so that every term of the step shows in D and W: two terms where the
step is below 0.03 / beta (FP64: 3e-4 / beta), four above, up to a widened fermi_lin.  The expected rows are the same Taylor
sum from the oracle's eigenpairs, at the step the call reports.  Bounds: FP32-class forms 6e-6 for D_c, four times the
1.3e-6 its rows show at 96 atoms, and 8e-6 for W_c (levels up to 1.3 Ha); FP64 5e-10, above the 1e-12 of its Ewald sums by
what a few dozen products and beta can make of it.  Each term is checked to be at least twice the bound.
"""
import numpy as np
import pytest

from oracle import density as odn
from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {0: (5e-10, 5e-10), 1: (6e-6, 8e-6), 4: (6e-6, 8e-6)}
TE = 30000.0
BETA = 1.0 / (3.166811563e-6 * TE)


@pytest.mark.parametrize("precision,shift,terms", [(0, 2.8e-4, 2), (0, 0.6, 4), (1, 2.8e-2, 2), (1, 0.6, 4),
                                                   (4, 2.8e-2, 2), (4, 0.6, 4)])
def test_rows_after_the_step(precision, shift, terms):
    from paper_2606_03140_gb300 import sedacs as S

    s = I.small_water_box(24, (29.97 * 24) ** (1 / 3), 724)
    m = I.default_model()
    n = I.random_charges(s.n_atoms, 6, 0.02)
    a = np.arange(s.n_atoms, dtype=np.int32)
    cores = [a[:30], a[30:]]                          # the subgraphs are the whole box, cores first
    ref = odn.density(s.R, s.species, s.box, m, n, cores, [a[30:], a[:30]], Te=TE)
    prm = S.sedacs_default_params(precision=precision, r_graph=30.0, Te=TE, fermi_lin=0.9)
    ctx = S.sedacs_create(s.species, s.box, m, prm)
    try:
        R = np.ascontiguousarray(s.R)
        S.sedacs_graph_build(ctx, R)
        S.sedacs_set_cores(ctx, cores)
        mu, _, _, _ = S.sedacs_subgraph_density(ctx, R, n, ref.mu - shift / BETA)
        info = S.sedacs_density_info(ctx)
        rows = [[S.sedacs_subgraph_matrix(ctx, i, which) for which in (4, 5)] for i in range(2)]
    finally:
        S.sedacs_destroy(ctx)
    x = BETA * info["dmu_linear"]
    limit = 3e-4 if precision == 0 else 3e-2
    assert info["passes"] == 1 and (x <= limit if terms == 2 else limit < x <= 0.9)
    for sg, (D, W) in zip(ref.subs, rows):
        f = odn.fermi(sg.eps - (mu - info["dmu_linear"]), BETA)
        t1 = f * (1 - f)
        t2 = t1 * (1 - 2 * f)
        t3 = t2 * (1 - 2 * f) - 2 * t1 * t1
        t4 = t3 * (1 - 2 * f) - 6 * t1 * t2
        parts = [f] + [c * t for c, t in zip((x, x**2 / 2, x**3 / 6, x**4 / 24), (t1, t2, t3, t4))][:terms]
        C, Cc = sg.C, sg.C[:int(sg.off[sg.n_core])]
        for got, level, tol in ((D, 1.0, TOL[precision][0]), (W, sg.eps, TOL[precision][1])):
            want = [2 * (Cc * (p * level)) @ C.T for p in parts]
            assert all(np.max(np.abs(p)) > 2 * tol for p in want)
            assert np.max(np.abs(got - sum(want))) < tol
