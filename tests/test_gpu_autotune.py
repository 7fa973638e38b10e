"""The launch-shape autotuner tries what can make a difference only: no parameter
without an effect on the call, no default against itself."""
import pytest

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_m,exact", [(0.0, False), (0.01, False), (0.0, True), (0.01, True)])
def test_candidates(d_m, exact):
    sc = G.scene_small((2, 2, 1), p=6, seed=3)
    sc.d_m = d_m
    eng = S.Stiv.for_scene(sc, pair_cap=64, contact_cap=1 << 15, exact_only=exact)
    ds = S.DeviceScene.from_scene(sc)
    eng.step(ds, grad=False)
    S.stiv_profile(eng.h, True)
    choice = eng.autotune(ds)
    runs = S.stiv_profile_read(eng.h)["narrow"][0]
    assert choice["fp64_blocks_per_sm"] in (0, 4, 8, 32) and choice["patch_blocks_per_sm"] in (0, 2, 4, 8)
    assert choice["piece_levels"] in ((0, 2, 3, 4) if d_m > 0 and not exact else (0,))
    assert choice["pieces_ctas_per_sm"] in ((0,) if exact else (0, 1, 2, 3, 4))
    # one step, two timings of the shapes at hand, then of each candidate, two runs
    # each: at most 3 (narrow) + 3 (FP64) + 3 (patch pairs), 4 (pieces), 3 (levels)
    most = 9 + (0 if exact else 4) + (3 if d_m > 0 and not exact else 0)
    assert 1 + 4 + 2 * 6 <= runs <= 1 + 4 + 2 * most
