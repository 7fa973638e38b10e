"""The mesh-fidelity tables of a handle, made on one stream and read on another
whose handle is the same number: the default stream of each thread.  The first
thread's stream is held up, so that the second would read tables that are not
written; and a third call rewrites them for another factor."""
import threading

import numpy as np
import pytest
import torch

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

pytestmark = pytest.mark.gpu

PER_THREAD = 2   # cudaStreamPerThread


def test_tables_across_threads():
    sc = G.two_vesicles(p=12, seed=3)
    ds = S.DeviceScene.from_scene(sc)
    eng, fresh = S.Stiv(), S.Stiv()
    eng.upsample(ds)
    want = {f: fresh.mesh_fidelity(ds, factor=f).cpu().numpy() for f in (3, 4)}
    torch.cuda.synchronize()
    got = {}

    def call(name, factor, hold):
        st = torch.cuda.ExternalStream(PER_THREAD)
        with torch.cuda.stream(st):
            if hold:
                torch.cuda._sleep(200_000_000)   # about a tenth of a second
            got[name] = eng.mesh_fidelity(ds, factor=factor, stream=st)

    for name, factor, hold in (("first", 4, True), ("second", 4, False), ("third", 3, False)):
        t = threading.Thread(target=call, args=(name, factor, hold))
        t.start()
        t.join()
    torch.cuda.synchronize()
    for name, factor in (("first", 4), ("second", 4), ("third", 3)):
        assert np.array_equal(got[name].cpu().numpy(), want[factor]), name
