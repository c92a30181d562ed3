"""Coulomb potential against the FP64 oracle at the edges of the reciprocal sums' blocks and of the cells.

Atom counts on either side of a staged run (64), a block of atoms (128) and an atom chunk (1,024), boxes with
unequal sides (k-rows of many lengths, odd and even row counts), and atoms crowded into a few cells.
"""
import numpy as np
import pytest

from oracle import ewald as oew
from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL_V = {0: 1e-9, 1: 1e-6}      # as for the other boxes: FP64, mixed


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_atoms,box,used", [
    (1, (9.0, 10.0, 11.0), 1.0), (3, (7.0, 12.0, 19.0), 1.0), (63, (9.5, 8.0, 8.0), 1.0), (65, (8.0, 9.0, 10.5), 1.0),
    (129, (11.0, 10.0, 13.0), 1.0), (1023, (28.0, 31.0, 45.5), 1.0), (1025, (47.0, 30.0, 28.5), 0.5)])
def test_potential(n_atoms, box, used, precision):
    from paper_2606_03140_gb300 import sedacs as S

    rng = np.random.default_rng(n_atoms)
    box = np.array(box)
    # jittered lattice points, so that no two atoms come near each other
    side = int(np.ceil(n_atoms ** (1 / 3)))
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)
    R = (rng.permutation(g)[:n_atoms] + rng.uniform(0.25, 0.75, (n_atoms, 3))) / side * box * used
    species = rng.integers(0, 3, n_atoms).astype(np.int32)
    m = I.default_model()
    q = rng.normal(0.0, 0.3, n_atoms)
    ref = oew.coulomb_potential(R, species, m.hubbard_u, box, q)
    ctx = S.sedacs_create(species, box, m, S.sedacs_default_params(precision=precision))
    try:
        V = S.sedacs_coulomb_potential(ctx, np.ascontiguousarray(R), q)
    finally:
        S.sedacs_destroy(ctx)
    assert np.max(np.abs(V - ref)) < TOL_V[precision]
