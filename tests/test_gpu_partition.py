"""Cores of the GPU bisection against the oracle's, exactly, on coordinates with many ties.

A cubic lattice (every plane holds atoms of equal coordinate, ranked by index), planes of more atoms than a
slice's ranking takes (the splits fall back to sorting), and a jittered box; partial last levels throughout.
"""
import numpy as np
import pytest

from oracle import graph as og
from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _lattice(nx, ny, nz, ax, ay, az):
    g = np.stack(np.meshgrid(np.arange(nx) * ax, np.arange(ny) * ay, np.arange(nz) * az, indexing="ij"), -1)
    return g.reshape(-1, 3) + 0.5, np.array([nx * ax, ny * ay, nz * az], dtype=np.float64)


CASES = {"cube": _lattice(11, 11, 11, 3.0, 3.0, 3.0), "planes": _lattice(4, 34, 34, 30.0, 2.0, 2.0),
         "jitter": (np.random.default_rng(5).uniform(-20.0, 60.0, (1237, 3)), np.array([31.0, 29.0, 37.0]))}


@pytest.mark.parametrize("core_size", [12, 32])
@pytest.mark.parametrize("name", list(CASES))
def test_cores_match_oracle(name, core_size):
    from paper_2606_03140_gb300 import sedacs as S
    R, box = CASES[name]
    R = np.ascontiguousarray(R[np.random.default_rng(9).permutation(len(R))])
    ctx = S.sedacs_create(np.full(len(R), I.H, np.int32), box, I.default_model(),
                          S.sedacs_default_params(core_size=core_size, r_graph=1.0))
    try:
        S.sedacs_graph_build(ctx, R)
        S.sedacs_partition(ctx, R)
        ptr, atoms, n_core = S.sedacs_parts_get(ctx)
    finally:
        S.sedacs_destroy(ctx)
    ref = og.rcb_partition(R, box, core_size)
    assert len(ref) == len(n_core)
    for i, c in enumerate(ref):
        assert list(atoms[ptr[i]:ptr[i] + n_core[i]]) == list(c)
