"""Chained Fermi-recursion products against the FP64 oracle at the edges of their tiles.

One subgraph holding the whole box, so that its orbital count sits on either side of the k-block (64)
and tile (128) boundaries and below one k-step; and one partition with subgraphs of very different sizes,
which finish their products at different times.  Bound: the 2e-5 e that the FP32-class forms 1 (two fp16
planes) and 4 (three bf16 planes) are held to at a chemical potential solved by each side.
"""
import numpy as np
import pytest

from oracle import density as odn
from oracle import graph as og
from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2606_03140_gb300 import sedacs
    return sedacs


def _charges(S, s, n, cores, precision, r_graph, Te):
    prm = S.sedacs_default_params(precision=precision, r_graph=r_graph, Te=Te)
    ctx = S.sedacs_create(s.species, s.box, I.default_model(), prm)
    try:
        R = np.ascontiguousarray(s.R)
        S.sedacs_graph_build(ctx, R)
        S.sedacs_set_cores(ctx, cores)
        mu, q, _, _ = S.sedacs_subgraph_density(ctx, R, n)
        # the same again from the mu of the first call: shifts at the kept stage and a second chain
        _, q2, _, _ = S.sedacs_subgraph_density(ctx, R, n, mu + 4e-3)
        return q, q2
    finally:
        S.sedacs_destroy(ctx)


# orbitals 6 per molecule: 60, 66, 126, 132, 192, 258, 384
@pytest.mark.parametrize("precision", [1, 4])
@pytest.mark.parametrize("n_water", [10, 11, 21, 22, 32, 43, 64])
def test_one_subgraph(S, n_water, precision):
    s = I.small_water_box(n_water, (29.97 * n_water) ** (1 / 3), 700 + n_water)
    n = I.random_charges(s.n_atoms, 5, 0.02)
    cores, halos = odn.full_partition(s.n_atoms)
    ref = odn.density(s.R, s.species, s.box, I.default_model(), n, cores, halos)
    for q in _charges(S, s, n, cores, precision, 3.0, 300.0):
        assert np.max(np.abs(q - ref.q)) < 2e-5


# Te 30,000 K needs few doublings (the kept stage is the first one)
@pytest.mark.parametrize("Te", [300.0, 30000.0])
@pytest.mark.parametrize("precision", [1, 4])
def test_uneven_subgraphs(S, precision, Te):
    s = I.small_water_box(43, (29.97 * 43) ** (1 / 3), 743)
    n = I.random_charges(s.n_atoms, 6, 0.02)
    cut = [0, 3, 6, 60, 75, s.n_atoms]
    cores = [np.arange(a, b, dtype=np.int32) for a, b in zip(cut[:-1], cut[1:])]
    rp, col = og.build_graph(s.R, s.box, 3.5)
    ref = odn.density(s.R, s.species, s.box, I.default_model(), n, cores, og.halos(rp, col, cores), Te=Te)
    for q in _charges(S, s, n, cores, precision, 3.5, Te):
        assert np.max(np.abs(q - ref.q)) < 2e-5
