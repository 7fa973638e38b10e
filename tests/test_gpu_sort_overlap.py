"""Sorting into arrays that overlap the input partly: the output keys lie over the
end of the input keys and over the input values, for every parity of the number
of digit passes, none (key_bits = 0, a copy) among them."""
import numpy as np
import pytest

from paper_1812_04719_gb300 import stiv as S

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 5000])
@pytest.mark.parametrize("bits", [0, 5, 12, 20])
@pytest.mark.parametrize("static", [False, True])
def test_output_over_the_input(n, bits, static):
    rng = np.random.default_rng(n + bits)
    k = rng.integers(0, 1 << 40, size=n, dtype=np.int64)
    v = rng.permutation(n).astype(np.int32)
    buf = torch.zeros(2 * n, dtype=torch.int64, device="cuda")   # keys, then values; the output keys from n / 2 on
    buf[:n] = torch.from_numpy(k).cuda()
    vals = buf[n:].view(torch.int32)[:n]
    vals.copy_(torch.from_numpy(v))
    ko = buf[n // 2:n // 2 + n]
    vo = torch.empty(n, dtype=torch.int32, device="cuda")
    args = (torch.cuda.current_stream().cuda_stream, n, bits, buf.data_ptr(), vals.data_ptr(), ko.data_ptr(),
            vo.data_ptr())
    if static:
        S.stiv_sort_pairs_static(*args)
    else:
        nb = S.stiv_sort_scratch_bytes(n)
        scratch = torch.empty(nb, dtype=torch.uint8, device="cuda")
        S.stiv_sort_pairs(*args, scratch.data_ptr(), nb)
    order = np.argsort(k & ((1 << bits) - 1), kind="stable")
    assert np.array_equal(ko.cpu().numpy(), k[order])
    assert np.array_equal(vo.cpu().numpy(), v[order])
