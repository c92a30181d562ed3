"""Forces after an accepted step of the chemical potential against the oracle, with two and with four terms.

D_c and the rows that W_c is formed from get the terms of the step's expansion; the starting guess decides how many.
Bounds: charges as in the 96-atom parity tests for each form (a potential solved by each side); forces 1e-7 Ha/A in
FP64 as there, and twice the 1e-3 of the largest force (0.05 Ha/A) that the FP32-class recursions leave.
"""
import numpy as np
import pytest

from oracle import density as odn
from oracle import graph as og
from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {0: (1e-8, 1e-7), 1: (2e-5, 1e-4), 4: (2e-5, 1e-4)}      # charges (e), forces (Ha/A)
BETA = 1.0 / (3.166811563e-6 * 300.0)


@pytest.mark.parametrize("precision", [0, 1, 4])
@pytest.mark.parametrize("shift", [2e-4, 1.2e-1])               # beta x (guess - solution)
def test_forces(precision, shift):
    from paper_2606_03140_gb300 import sedacs as S

    s = I.small_water_box(24, (29.97 * 24) ** (1 / 3), 724)
    m = I.default_model()
    R = np.ascontiguousarray(s.R)
    n = I.random_charges(s.n_atoms, 6, 0.02)
    cut = [0, 5, 30, s.n_atoms]
    cores = [np.arange(a, b, dtype=np.int32) for a, b in zip(cut[:-1], cut[1:])]
    rp, col = og.build_graph(s.R, s.box, 3.5)
    ref = odn.density(s.R, s.species, s.box, m, n, cores, og.halos(rp, col, cores))
    Fref = odn.forces(ref, n, s.R, s.species, s.box, m)
    ctx = S.sedacs_create(s.species, s.box, m, S.sedacs_default_params(precision=precision, r_graph=3.5))
    try:
        S.sedacs_graph_build(ctx, R)
        S.sedacs_set_cores(ctx, cores)
        _, q, _, _ = S.sedacs_subgraph_density(ctx, R, n, ref.mu + shift / BETA)
        F = S.sedacs_forces(ctx, s.n_atoms)
    finally:
        S.sedacs_destroy(ctx)
    assert np.max(np.abs(q - ref.q)) < TOL[precision][0]
    assert np.max(np.abs(F - Fref)) < TOL[precision][1]
