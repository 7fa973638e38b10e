"""The count of patch pairs where a patch touches both poles (order 1): its two
halves are examined apart, but it is one patch."""
import pytest

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S
from tests.gpu_run import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [S.STIV_FP64, S.STIV_MIXED])
def test_one_patch_per_vesicle(precision):
    g = run_gpu(G.two_vesicles(p=1, seed=1, gap=-0.3, approach=0.5), precision=precision, grad=False)
    assert g["counts"][S.C_VF] + g["counts"][S.C_EE] > 0
    assert g["counts"][S.C_PAIRS] == 1 and g["counts"][S.C_PATCH] == 1


def test_orders_one_and_two():
    """Order 1 has one patch of 2 x 4 quads, order 2 two bands of two: at most 4
    patch pairs between them, and each vesicle pair with primitive pairs has one."""
    a, b = G.two_vesicles(p=1, seed=1, gap=-0.3, approach=0.5), G.two_vesicles(p=2, seed=1, gap=-0.3, approach=0.5)
    sc = G._pack("1 and 2", [1, 2], [a.coef_of(0), b.coef_of(1)], a.L, a.centers)
    c = run_gpu(sc, grad=False)["counts"]
    assert c[S.C_PRIM] > 0 and 1 <= c[S.C_PATCH] <= 4
