"""The mesh-fidelity tables that a handle keeps: calls that change the factor, the
largest order, the vesicle count (one chunk of rings per CTA or many) and the
stream give the results of a fresh handle bit for bit."""
import numpy as np
import pytest
import torch

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

pytestmark = pytest.mark.gpu


def fidelity(eng, ds, factor, stream=None):
    e = eng.mesh_fidelity(ds, factor=factor, stream=stream)
    torch.cuda.synchronize()
    return e.cpu().numpy().view(np.int64)


def test_kept_tables_follow_the_call():
    one = G.two_vesicles(p=7, seed=3)
    many = G.lattice_scene("fid", (6, 6, 4), 0.4, [5 + 3 * (k % 2) for k in range(288)], 4, tilt_deg=0.0,
                           trans_amp=0.1, rot_deg=1.0, pert=0.02, cubic=False, periodic=False)
    side = torch.cuda.Stream()
    for prec in (S.STIV_FP64, S.STIV_MIXED):
        kept = S.Stiv(precision=prec)
        scenes = []
        for sc in (one, many):
            ds = S.DeviceScene.from_scene(sc, precision=prec)
            kept.upsample(ds)
            scenes.append(ds)
        torch.cuda.synchronize()
        for k, factor, stream in ((0, 4, None), (0, 4, None), (0, 2, None), (1, 2, None), (1, 4, side), (0, 4, side),
                                  (0, 8, None), (1, 1, None)):
            fresh = S.Stiv(precision=prec)
            got = fidelity(kept, scenes[k], factor, stream)
            assert np.array_equal(got, fidelity(fresh, scenes[k], factor)), (k, factor)
            assert factor == 1 or np.all(got > 0)   # factor 1: the mesh vertices themselves, rounding only
