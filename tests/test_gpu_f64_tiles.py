"""FP64 products (form 0) against the oracle at the edges of their tiles and of the warps' blocks in them.

One subgraph holding the whole box, its orbital count (6 per molecule) on either side of the blocks (16), the
tiles (32) and the matrix padding (128), and a partition whose core rows end inside a block.  Bounds: the 1e-8 e
that form 0 is held to at a chemical potential solved by each side, and without temperature at a given one.
"""
import numpy as np
import pytest

from oracle import density as odn
from oracle import graph as og
from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _charges(s, n, cores, r_graph, Te=300.0, mu=None):
    from paper_2606_03140_gb300 import sedacs as S

    prm = S.sedacs_default_params(precision=0, r_graph=r_graph, Te=Te)
    ctx = S.sedacs_create(s.species, s.box, I.default_model(), prm)
    try:
        R = np.ascontiguousarray(s.R)
        S.sedacs_graph_build(ctx, R)
        S.sedacs_set_cores(ctx, cores)
        return S.sedacs_subgraph_density(ctx, R, n, **({} if mu is None else {"mu": mu}))[1]
    finally:
        S.sedacs_destroy(ctx)


# orbitals: 48, 60, 66, 96, 126, 132
@pytest.mark.parametrize("n_water", [8, 10, 11, 16, 21, 22])
def test_one_subgraph(n_water):
    s = I.small_water_box(n_water, (29.97 * max(n_water, 10)) ** (1 / 3), 700 + n_water)
    n = I.random_charges(s.n_atoms, 5, 0.02)
    cores, _ = odn.full_partition(s.n_atoms)
    ref = odn.density(s.R, s.species, s.box, I.default_model(), n, *odn.full_partition(s.n_atoms))
    assert np.max(np.abs(_charges(s, n, cores, 3.0) - ref.q)) < 1e-8
    # Te = 0: the traces of the diagonal tiles steer the recursion; mu in the widest gap, more than 30 kT from levels
    e = np.sort(ref.subs[0].eps)
    k = np.argmax(np.diff(e))
    assert e[k + 1] - e[k] > 0.06
    mu = 0.5 * (e[k] + e[k + 1])
    gap = odn.density(s.R, s.species, s.box, I.default_model(), n, *odn.full_partition(s.n_atoms), mu=mu)
    assert np.max(np.abs(_charges(s, n, cores, 3.0, 0.0, mu) - gap.q)) < 1e-8


def test_uneven_subgraphs():
    s = I.small_water_box(43, (29.97 * 43) ** (1 / 3), 743)
    n = I.random_charges(s.n_atoms, 6, 0.02)
    cut = [0, 3, 6, 60, 75, s.n_atoms]
    cores = [np.arange(a, b, dtype=np.int32) for a, b in zip(cut[:-1], cut[1:])]
    rp, col = og.build_graph(s.R, s.box, 3.5)
    ref = odn.density(s.R, s.species, s.box, I.default_model(), n, cores, og.halos(rp, col, cores))
    assert np.max(np.abs(_charges(s, n, cores, 3.5) - ref.q)) < 1e-8
