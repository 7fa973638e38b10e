"""A captured step whose handle's scratch grows in between: the small step is
captured, a larger eager one grows the scratch, and the small one, with the same
arguments, gives a fresh handle's results."""
import numpy as np
import pytest
import torch

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

pytestmark = pytest.mark.gpu

KEYS = ("i", "j", "shift", "pair", "type", "a", "b", "tau", "w", "V", "V_pair", "grad", "gves", "gvid")


def snapshot(r, ds):
    out = {k: r[k].cpu().numpy().copy() for k in KEYS}
    out["counts"] = r["counts"].copy()
    out["verts"] = ds.verts.cpu().numpy().copy()
    return out


@pytest.mark.parametrize("precision", [S.STIV_FP64, S.STIV_MIXED])
@pytest.mark.parametrize("larger", ["step", "upsample"])
def test_graph_follows_the_scratch(precision, larger):
    kw = dict(precision=precision, pair_cap=1024, contact_cap=1 << 16)
    a = G.scene_small((2, 1, 1), p=4, seed=3)
    big = G.lattice_scene("big", (4, 4, 2), 0.4, [8] * 64, 4, tilt_deg=0.0, trans_amp=0.2, rot_deg=1.0, pert=0.02,
                          cubic=False, periodic=False)
    st = torch.cuda.Stream()
    dsa, dsb = S.DeviceScene.from_scene(a, precision=precision), S.DeviceScene.from_scene(big, precision=precision)
    torch.cuda.synchronize()
    fresh = S.Stiv(box_L=tuple(a.L), eps=a.eps, dt=a.dt, **kw)
    want = snapshot(fresh.step(dsa, grad=True), dsa)
    eng = S.Stiv(box_L=tuple(a.L), eps=a.eps, dt=a.dt, **kw)
    for _ in range(2):                  # captured, replayed
        r = eng.step(dsa, grad=True, use_graph=True, stream=st)
    if larger == "step":
        eng.step(dsb, grad=True, stream=st)
    else:                               # only the mixed form's synthesis has scratch of its own
        eng.upsample(dsb, stream=st)
    for _ in range(2):
        dsa.verts.zero_()
        torch.cuda.synchronize()
        got = snapshot(eng.step(dsa, grad=True, use_graph=True, stream=st), dsa)
        for k, v in want.items():
            assert np.array_equal(got[k], v), k
