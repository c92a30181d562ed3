"""Device memory of a context against the matrices a density call works on.

A context holds, per subgraph, 17 square matrices and 12 sets of core rows (matrices and rows that are operands of the
FP32-class products with three 16-bit planes beside the FP32 master: 10 bytes an element, others 4), and a quarter more so that
a growing graph does not reallocate.  The rest here is the blocks of the pairs (about 140,000 at 160 bytes, 22 MB) and a
few MB of atom, Ewald and layout tables.  The bound of 60 MB for it lies halfway to four further sets of core rows (120 MB):
the largest box that fits the GPU is decided by the matrices.
"""
import numpy as np
import pytest

from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _density(S, s, r_graph):
    """Free memory and subgraphs of a context that has computed a density."""
    import torch

    R = np.ascontiguousarray(s.R)
    ctx = S.sedacs_create(s.species, s.box, I.default_model(), S.sedacs_default_params(precision=1, r_graph=r_graph))
    try:
        S.sedacs_graph_build(ctx, R)
        S.sedacs_partition(ctx, R)
        S.sedacs_subgraph_density(ctx, R, np.ascontiguousarray(I.random_charges(s.n_atoms, 5, 0.02)))
        return torch.cuda.mem_get_info()[0], S.sedacs_parts_get(ctx)
    finally:
        S.sedacs_destroy(ctx)


def test_arena_holds_no_more_than_its_matrices():
    import torch
    from paper_2606_03140_gb300 import sedacs as S

    _density(S, I.workload("water96"), 3.0)            # code and local memory of the kernels are loaded
    s = I.small_water_box(511, (29.97 * 511) ** (1 / 3), 511)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    left, (ptr, atoms, n_core) = _density(S, s, 4.0)
    orb = np.asarray(I.default_model().n_orb)[s.species]
    pad = lambda n: max(128, -(-int(n) // 128) * 128)
    square = rows = 0
    for i, (a, b) in enumerate(zip(ptr[:-1], ptr[1:])):
        n, c = pad(orb[atoms[a:b]].sum()), pad(orb[atoms[a:a + n_core[i]]].sum())
        square += n * n
        rows += c * n
    arena = 1.25 * (17 * 10 * square + (6 * 10 + 6 * 4) * rows)
    assert 1.25 * 4 * 10 * rows > 119e6                # what the bound below can tell apart
    assert free - left < arena + 60e6
