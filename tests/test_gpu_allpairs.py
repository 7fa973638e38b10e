"""Candidate vesicle pairs by the all-pairs box test and by the Morton grid, on
both sides of the vesicle count where the library changes over (8192), against
the oracle's all-pairs box test: the same pairs and shifts in the same order.
Small and ragged counts, rows with more hits than a unit keeps, periodic boxes
and free space, vesicles of very different size."""
import math

import numpy as np
import pytest

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S
from tests.gpu_run import gpu_pairs_rows, run_gpu_on, verts_list
from tests.oracle_pool import oracle_vertices

pytestmark = pytest.mark.gpu


def spheres(n, L, radii, seed):
    """n spheres of order 1 at random places of a cube (L = 0: of side 10, free
    space), each moved by a small step."""
    rng = np.random.default_rng(seed)
    side = L if L > 0 else 10.0
    c = rng.uniform(0, side, size=(n, 3))
    r = np.exp(rng.uniform(math.log(radii[0]), math.log(radii[1]), size=n))
    step = rng.normal(size=(n, 3)) * 0.2 * radii[0]
    coefs = [np.stack([G.ellipsoid_coef(1, c[k], r[k] * np.eye(3)), G.ellipsoid_coef(1, c[k] + step[k], r[k] * np.eye(3))])
             for k in range(n)]
    return G._pack("spheres", [1] * n, coefs, [L] * 3, c)


@pytest.mark.parametrize("n,L,radii", [(2, 0.0, (3.0, 4.0)), (3, 40.0, (5.0, 9.0)), (33, 20.0, (1.0, 3.0)),
                                       (513, 30.0, (0.5, 3.0)), (600, 24.0, (4.0, 5.0)), (1500, 0.0, (0.1, 0.6)),
                                       (8192, 60.0, (0.2, 0.8)), (8193, 60.0, (0.2, 0.8))])
def test_candidate_pairs_match_all_pairs(orc, n, L, radii):
    sc = spheres(n, L, radii, seed=n)
    X = oracle_vertices(sc)
    g = run_gpu_on(sc, X, grad=False, pair_cap=64 * n, contact_cap=1 << 18)
    boxes = np.stack([orc.vesicle_box(x, 0.0) for x in verts_list(sc, X)])
    pairs = orc.candidate_pairs(boxes, sc.L)
    assert n < 500 or len(pairs) > n // 16
    assert np.array_equal(gpu_pairs_rows(g), pairs)
