"""Graph edges at the cutoff, whole numbers compared with the oracle.

Lattices whose neighbours lie at the cutoff to within the rounding of the coordinates, atoms moved by whole boxes
(so that FP32 coordinates are far too coarse), and positions on the faces of the box, where both images are equally
far: the pairs whose distance the FP32 test must leave to the FP64 one.
"""
import numpy as np
import pytest

from oracle import graph as og
from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jitter", [0.0, 1e-14, 1e-7, 1e-4])
@pytest.mark.parametrize("boxes", [0, 3, 20000])
@pytest.mark.parametrize("cells", [2, 3, 10])           # lattice cells per axis: image loop, smallest and larger grid
def test_edges(cells, boxes, jitter):
    from paper_2606_03140_gb300 import sedacs as S

    r = 6.0
    box = np.array([r, r, r * 1.01]) * (cells + (cells > 2) * 1e-6)
    rng = np.random.default_rng(cells * 7 + boxes)
    g = np.stack(np.meshgrid(*[np.arange(cells)] * 3, indexing="ij"), -1).reshape(-1, 3)
    R = g * np.array([r, r, r * 1.01]) + rng.integers(-boxes, boxes + 1, g.shape) * box
    R = np.ascontiguousarray(R + jitter * rng.standard_normal(R.shape))
    species = np.zeros(len(R), np.int32)
    ptr, col = og.build_graph(R, box, r)
    ctx = S.sedacs_create(species, box, I.default_model(), S.sedacs_default_params(precision=1, r_graph=r))
    try:
        nnz = S.sedacs_graph_build(ctx, R)
        p, c = S.sedacs_graph_get(ctx, len(R), nnz)
    finally:
        S.sedacs_destroy(ctx)
    assert np.array_equal(p, ptr) and np.array_equal(c, col)
