"""Rounding of the learned kernel's layers, whose corrections are small against the residual they are added to.

The parameters and vectors are FP32 numbers, so that what is left against the FP64 oracle is the layers' own rounding.
Emulated in FP32 on the CPU for these seeds: 0.7e-7 and 1.0e-7 of the largest G(y) where the corrections are summed
from zero and added once, 5e-7 and 14e-7 where they are summed on top of the residual; gradients of the embedding
1.0e-7 and 0.8e-7 against 4.0e-7 and 5.7e-7.  Bounds: between the two, 3e-7 and 2.5e-7.
"""
import numpy as np
import pytest

from oracle import gnn as ognn
from oracle import graph as og
from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [0, 1])
def test_corrections_are_added_once(seed):
    from paper_2606_03140_gb300 import sedacs as S

    s = I.workload("water96")
    f32 = lambda x: x.astype(np.float32).astype(np.float64)
    d = ognn.unpack(ognn.init_params(seed))
    for l in range(ognn.NLAYER):
        d["A"][l], d["B"][l] = 0.1 * d["A"][l], 0.1 * d["B"][l]
    p = f32(ognn.pack(d))
    rng = np.random.default_rng(seed)
    y, gu = f32(rng.standard_normal(96)), f32(rng.standard_normal(96))
    rp, col = og.build_graph(s.R, s.box, 3.0)
    edges = ognn.edges_from_csr(rp, col, s.R, s.box)
    G_ref = ognn.forward(p, y, s.species, edges, 0.5) + 0.5 * y
    g_ref = ognn.backward(p, y, s.species, edges, 0.5, gu)[:192]
    ctx = S.sedacs_create(s.species, s.box, I.default_model(), S.sedacs_default_params(precision=1, c_k0=0.5))
    try:
        S.sedacs_graph_build(ctx, np.ascontiguousarray(s.R))
        S.sedacs_gnn_set_params(ctx, p)
        G = S.sedacs_gnn_apply(ctx, y) + 0.5 * y
        g = S.sedacs_gnn_param_grad(ctx, y, gu)[:192]
    finally:
        S.sedacs_destroy(ctx)
    assert np.max(np.abs(G - G_ref)) < 3e-7 * np.max(np.abs(G_ref))
    assert np.max(np.abs(g - g_ref)) < 2.5e-7 * np.max(np.abs(g_ref))
