"""The 16-bit histogram of the QCrank decode at its edges: the shot count where
it takes over, chunk remainders, counters that fill (every shot at one
address), and the largest table it holds."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2504_03967_gb300 as S
from oracle import qcrank_ref as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a,d,shots", [(14, 6, 1245100), (14, 6, 1400000), (15, 2, 65535 * 20), (13, 12, 2000001)])
@pytest.mark.parametrize("same", [False, True], ids=["random", "one-address"])
def test_sixteen_bit_histogram(a, d, shots, same):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(a + d)
    x = rng.integers(0, 1 << (a + d + 3), size=shots, dtype=np.int64)
    if same:
        x[:] = (1 << (a + d)) - 1
    dx = torch.from_numpy(x).cuda()
    counts = torch.full((1 << a,), 7, dtype=torch.int64, device="cuda")
    ones = torch.full(((1 << a) * d,), 7, dtype=torch.int64, device="cuda")
    pixels = torch.zeros((1 << a) * d, dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    S.sv_qcrank_decode_device(dx.data_ptr(), shots, a, d, counts.data_ptr(), ones.data_ptr(), pixels.data_ptr(), st)
    torch.cuda.synchronize()
    _, wc, wo = Q.decode(x.astype(np.uint64), a, d)
    assert np.array_equal(counts.cpu().numpy(), wc)
    assert np.array_equal(ones.cpu().numpy().reshape(1 << a, d), wo)
