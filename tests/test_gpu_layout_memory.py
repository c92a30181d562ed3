"""A context whose new subgraphs do not fit the device: refused calls, then other cores and the results of before."""
import numpy as np
import pytest

from paper_2606_03140_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_cores_that_do_not_fit(precision):
    from paper_2606_03140_gb300 import sedacs as S

    # water molecules on a grid: 36,000 orbitals, whose matrices in one subgraph take 300 GB and more
    side, a = (20, 20, 15), 3.6
    g = np.stack(np.meshgrid(*[np.arange(k) for k in side], indexing="ij"), -1).reshape(-1, 1, 3) * a
    R = np.ascontiguousarray((g + np.array([[0, 0, 0], [0.76, 0.59, 0], [-0.76, 0.59, 0]])).reshape(-1, 3))
    species = np.tile([I.O, I.H, I.H], len(g)).astype(np.int32)
    n_at = len(R)
    small = [np.arange(i, min(n_at, i + 96), dtype=np.int32) for i in range(0, n_at, 96)]
    n = np.ascontiguousarray(np.tile([-0.3, 0.15, 0.15], len(g)))
    ctx = S.sedacs_create(species, np.array(side) * a, I.default_model(),
                          S.sedacs_default_params(precision=precision, r_graph=2.0, Te=3000.0))
    try:
        S.sedacs_graph_build(ctx, R)
        S.sedacs_set_cores(ctx, small)
        mu, q, _, _ = S.sedacs_subgraph_density(ctx, R, n)
        with pytest.raises(S.SedacsError) as e:
            S.sedacs_set_cores(ctx, [np.arange(n_at, dtype=np.int32)])
        assert e.value.status == 2                     # SEDACS_ENOMEM
        for call in (lambda: S.sedacs_subgraph_density(ctx, R, n), lambda: S.sedacs_forces(ctx, n_at),
                     lambda: S.sedacs_charge_response(ctx, n), lambda: S.sedacs_subgraph_matrix(ctx, 0, 0)):
            with pytest.raises(S.SedacsError) as e:
                call()
            assert e.value.status == 1                 # SEDACS_EINVAL
        S.sedacs_set_cores(ctx, small)
        mu2, q2, _, _ = S.sedacs_subgraph_density(ctx, R, n)
    finally:
        S.sedacs_destroy(ctx)
    assert mu2 == mu and np.array_equal(q2, q)
