"""A call that CUDA refuses on the host is reported once: PyTorch's next launch and
the next good call see nothing of it."""
import numpy as np
import pytest
import torch

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

pytestmark = pytest.mark.gpu

LEGACY_STREAM = 1   # cudaStreamLegacy, which CUDA does not let be captured


def test_refused_capture_is_reported_once():
    sc = G.scene_pair()
    eng = S.Stiv.for_scene(sc, pair_cap=16, contact_cap=1024)
    ds = S.DeviceScene.from_scene(sc)
    want = eng.step(ds, grad=True)["tau"].cpu().numpy().copy()
    b = eng.buf
    with pytest.raises(S.StivError) as e:
        S.stiv_step(eng.h, LEGACY_STREAM, True, ds.n, ds.p_max, S._ptr(ds.p), S._ptr(ds.coef_off), S._ptr(ds.coef),
                    S._ptr(ds.vert_off), S._ptr(ds.verts), b.pairs_struct(), b.contacts_struct(), S._ptr(b.counts),
                    S._ptr(b.Vc), S._ptr(b.Vp), S._ptr(b.grad), S._ptr(b.gves), S._ptr(b.gvid))
    # (nothing between: a good call of the runtime may take the pending error off)
    assert float((torch.ones(4, device="cuda") * 2).sum()) == 8.0
    assert e.value.status == S.STIV_ERR_CUDA and S.lib().stiv_last_cuda_error(eng.h) != 0
    got = eng.step(ds, grad=True)["tau"].cpu().numpy()
    assert np.array_equal(got.view(np.int64), want.view(np.int64))
