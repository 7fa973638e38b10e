"""Handles of different largest orders in concurrent threads, each on its own stream:
the kernels' limits of shared memory belong to the device, so no thread's call may
lower what another's is about to use."""
import threading

import numpy as np
import pytest
import torch

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

pytestmark = pytest.mark.gpu


def test_concurrent_calls_of_different_orders():
    orders = (4, 8, 22, 32)
    n = 100                 # few vesicles: one field a CTA; more than 75: three
    jobs = []
    for p in orders:
        a = G.two_vesicles(p=p, seed=1)
        sc = G._pack(f"{p}", [p] * n, [a.coef_of(k % 2) for k in range(n)], np.zeros(3), np.zeros((n, 3)))
        pair = G.two_vesicles(p=p, seed=1)
        ds, dp = S.DeviceScene.from_scene(sc), S.DeviceScene.from_scene(pair)
        eng = S.Stiv(pair_cap=16, contact_cap=1 << 14)
        gX, gc = torch.ones(dp.verts.numel(), dtype=torch.float64, device="cuda"), torch.zeros_like(dp.coef)
        jobs.append((eng, ds, dp, gX, gc, torch.cuda.Stream()))
    torch.cuda.synchronize()
    errors = []
    gate = threading.Barrier(len(jobs))

    def work(eng, ds, dp, gX, gc, st):
        q = st.cuda_stream
        b = eng._buffers(False)
        gate.wait()
        for k in range(150):
            try:
                eng.upsample(ds, stream=st)
                eng.upsample(dp, stream=st)
                S.stiv_grad_to_coef(eng.h, q, dp.n, dp.p_max, S._ptr(dp.p), S._ptr(dp.coef_off), S._ptr(dp.vert_off),
                                    S._ptr(gX), S._ptr(gc))
                S.stiv_detect(eng.h, q, dp.n, dp.p_max, S._ptr(dp.p), S._ptr(dp.vert_off), S._ptr(dp.verts),
                              b.pairs_struct(), b.contacts_struct(), S._ptr(b.counts))
            except S.StivError as e:
                errors.append((dp.p_max, k, str(e)))
                return

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
