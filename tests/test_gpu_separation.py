"""Stage 1's slot masks and stage 3a's separation certificate change no result:
with and without the FP32 rejection (exact_only) the contact lists, times,
weights and the counts of pairs tested and degenerate agree bit for bit.  The
scenes put the certificate where it could go wrong: unperturbed vesicles with
parallel axes (edges that stay parallel, primitives coplanar throughout, exact
zeros in the polynomial), patches with both poles (p = 1), odd orders, and a
suspension far from the origin, where the FP64 positions themselves are
coarse."""
import math

import numpy as np
import pytest

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S
from tests.gpu_run import run_gpu

pytestmark = pytest.mark.gpu


def aligned(p, pert=0.0, trans=0.5, flow=0.0, shift=0.0):
    """3 x 3 x 2 staggered vesicles in free space, long axes along z."""
    ps = [p] * 36 if isinstance(p, int) else [p[k % len(p)] for k in range(36)]
    sc = G.lattice_scene("aligned", (3, 3, 2), 0.6, ps, 11, tilt_deg=0.0, trans_amp=trans, rot_deg=0.0, pert=pert,
                         shape_amp=0.0, flow_amp=flow, cubic=False, periodic=False)
    for v in range(sc.n):
        sc.coef_of(v)[:, :, 0] += math.sqrt(4 * math.pi) * shift
    return sc


@pytest.mark.parametrize("precision", [S.STIV_FP64, S.STIV_MIXED])
@pytest.mark.parametrize("d_m", [0.0, 0.03])
@pytest.mark.parametrize("name,kw", [("p1", dict(p=1)), ("p1_perturbed_flow", dict(p=(1, 2), flow=2.0)),
                                     ("p5_aligned", dict(p=5)), ("p7_mixed", dict(p=(3, 7), pert=0.02, flow=2.0)),
                                     ("p6_far", dict(p=6, pert=0.02, shift=3000.0)), ("p6_still", dict(p=6, trans=0.0))])
def test_rejection_is_exact(name, kw, d_m, precision):
    import dataclasses
    sc = dataclasses.replace(aligned(**kw), d_m=d_m)
    run = {}
    for exact in (False, True):
        eng = S.Stiv.for_scene(sc, precision=precision, pair_cap=1024, contact_cap=1 << 17, exact_only=exact)
        run[exact] = run_gpu(sc, precision=precision, eng=eng)
    f, x = run[False], run[True]
    assert x["counts"][S.C_PRIM] > 500
    for k in ("i", "j", "shift", "pair", "type", "a", "b"):
        assert np.array_equal(f[k], x[k]), k
    assert np.array_equal(f["tau"].view(np.int64), x["tau"].view(np.int64))
    assert np.array_equal(f["w"].view(np.int64), x["w"].view(np.int64))
    for c in (S.C_PAIRS, S.C_PRIM, S.C_VF, S.C_EE, S.C_CPAIRS, S.C_DEGEN):
        assert f["counts"][c] == x["counts"][c], c
