"""<Z_i> of complex64 states: sums over blocks keep what FP64 holds, and every
index bit of the block records is summed with its own records."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2504_03967_gb300 as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [13, 14, 18])
def test_small_masses_beside_a_large_one(n):
    """One amplitude of mass 1 + 2^-11 + 2^-24 and seven of 2^-49, each in its own
    block of 1024, qubits 0..9 set in all of them: every sum is exact in FP64,
    so <Z_i> = -S exactly."""
    v = np.zeros(1 << n, np.complex64)
    v[1023] = 1 + 2.0 ** -12
    for b in range(1, 8):
        v[1024 * b + 1023] = 2.0 ** -25 * (1 + 1j)
    total = (1 + 2.0 ** -12) ** 2 + 7 * 2.0 ** -49
    h = S.sv_alloc(n, S.C64)
    try:
        S.sv_load_state(h, v)
        _, ez = S.sv_measure(h, 100, 1)
        assert (S.sv_expect_z(h) == ez).all()
        assert np.abs(ez[:10] + total).max() <= 2.0 ** -51
    finally:
        S.sv_free(h)


@pytest.mark.parametrize("dtype,n", [(S.C64, 27), (S.C64, 28), (S.C128, 27)])
def test_every_index_bit(dtype, n):
    """A product state whose qubits all have different <Z_i>: 2^(n-10) block
    records, more than 256 per CTA."""
    torch = pytest.importorskip("torch")
    p1 = 0.05 + 0.9 * np.random.default_rng(n).permutation(n) / n
    amp = torch.ones(1, dtype=torch.float64, device="cuda")
    for p in p1:
        amp = torch.cat([amp * np.sqrt(1.0 - p), amp * np.sqrt(p)])
    state = amp.to(torch.complex64 if dtype == S.C64 else torch.complex128)
    del amp
    h = S.sv_attach(n, dtype, state.data_ptr(), torch.cuda.current_stream().cuda_stream)
    try:
        ez = S.sv_expect_z(h)
        # complex64: the amplitudes' rounding; independent over 2^n of them
        assert np.abs(ez - (1.0 - 2.0 * p1)).max() <= (2e-7 if dtype == S.C64 else 1e-12)
    finally:
        S.sv_free(h)
