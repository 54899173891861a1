"""The samplers' short cuts (CDF table for many shots, quarter totals for few
shots on a large state) give the outcome of the sampling rule, at the sizes
where their choice or their geometry changes."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2504_03967_gb300 as S
import workloads as W
from tests.gpu_util import BAND, compare_samples

pytestmark = pytest.mark.gpu


def _state(kind, n, seed):
    if kind == "random":
        return W.random_state(n, seed)
    v = np.zeros(1 << n, np.complex128)
    if kind == "basis":
        v[(1 << n) - 1] = 1.0
    else:  # "sparse": a few amplitudes, at both ends of blocks and quarters, the rest exactly zero
        at = [0, 31, 32, 255, 256, 767, 768, 1023, (1 << n) - 1024, (1 << n) - 1]
        v[at] = np.exp(1j * np.arange(len(at))) / np.sqrt(len(at))
    return v


def _cdf(h):
    # the rule applies to the state as stored (complex64 rounding included)
    a = S.sv_store_state(h).astype(np.complex128)
    return oracle.cdf(oracle.probs(a))


@pytest.mark.parametrize("dtype", [S.C64, S.C128])
@pytest.mark.parametrize("n", [10, 11, 16])
@pytest.mark.parametrize("kind", ["random", "basis", "sparse"])
def test_many_shots(dtype, n, kind):
    N = 1 << n
    h = S.sv_alloc(n, dtype)
    try:
        S.sv_load_state(h, _state(kind, n, n))
        cdf = _cdf(h)
        for shots in (N // 4 - 1, N // 4, N // 4 + 3, N, 3 * N + 1):  # both sides of the rule, every remainder of 4
            u = W.uniforms(shots, shots)
            u[:2] = 0.0, 1.0 - 2.0 ** -53
            compare_samples(S.sv_sample_uniforms(h, u), u, cdf, BAND)
    finally:
        S.sv_free(h)


@pytest.mark.parametrize("dtype", [S.C64, S.C128])
def test_many_shots_relabelled(dtype):
    n = 12
    h = S.sv_alloc(n, dtype)
    try:
        S.sv_init_basis(h, 0)
        S.sv_apply_circuit(h, np.concatenate([W.random_u3_cx(n, 2, 5), W.qft(n)]), relabel=1)
        assert S.sv_qubit_map(h) != list(range(n))
        cdf = _cdf(h)
        u = W.uniforms(2 << n, 9)
        compare_samples(S.sv_sample_uniforms(h, u), u, cdf, BAND)
    finally:
        S.sv_free(h)


@pytest.mark.parametrize("n", [9, 10, 11, 18])
@pytest.mark.parametrize("kind", ["random", "basis", "sparse"])
@pytest.mark.parametrize("scale", [1.0, 3e-13])
def test_shots_and_expz_together(n, kind, scale):
    if kind == "sparse" and n < 11:
        pytest.skip("needs more than one block")
    h = S.sv_alloc(n, S.C64)
    try:
        S.sv_load_state(h, scale * _state(kind, n, n))
        cdf = _cdf(h)
        samp, ez = S.sv_measure(h, 3001, 7)
        raw = np.random.Philox(key=7, counter=2 ** 256 - 1).random_raw(3001)
        u = (raw >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
        compare_samples(samp, u, cdf, BAND * scale * scale)
        p = np.diff(cdf, prepend=0.0)
        x = np.arange(1 << n)
        want = [p.sum() - 2.0 * p[(x >> q) & 1 == 1].sum() for q in range(n)]
        assert np.abs(ez - want).max() <= 1e-12 * cdf[-1]
    finally:
        S.sv_free(h)


@pytest.mark.parametrize("scale", [1e-149, 1e-141, 1e-139, 1e149])
def test_many_shots_far_from_unit_norm(scale):
    """Totals where 2^53 / S leaves the double range, and both sides of the line
    at which the table is no longer used."""
    n = 10
    h = S.sv_alloc(n, S.C128)
    try:
        S.sv_load_state(h, scale * W.random_state(n, 5))
        cdf = _cdf(h)
        u = W.uniforms(1 << 16, 6)
        # (the rule and its restatement add 2^n FP64 terms in different orders)
        compare_samples(S.sv_sample_uniforms(h, u), u, cdf, cdf[-1] * 2.0 ** (n - 52))
    finally:
        S.sv_free(h)


@pytest.mark.parametrize("dtype", [S.C64, S.C128])
@pytest.mark.parametrize("n,shots", [(10, 2 ** 15 - 1), (10, 2 ** 15), (10, 2 ** 15 + 3), (12, 40001), (16, 2 ** 15), (18, 2 ** 15),
                                     (19, 2 ** 19 // 12 - 1), (19, 2 ** 19 // 12), (19, 2 ** 19 // 12 + 2)])
@pytest.mark.parametrize("relabel", [0, 1])
def test_table_line(dtype, n, shots, relabel):
    """Both sides of the shot counts at which the CDF table takes over."""
    h = S.sv_alloc(n, dtype)
    try:
        S.sv_init_basis(h, 0)
        S.sv_apply_circuit(h, np.concatenate([W.random_u3_cx(n, 2, 5), W.qft(n)]), relabel=relabel)
        assert (S.sv_qubit_map(h) != list(range(n))) == bool(relabel)
        cdf = _cdf(h)
        u = W.uniforms(shots, 9)
        u[:2] = 0.0, 1.0 - 2.0 ** -53
        compare_samples(S.sv_sample_uniforms(h, u), u, cdf, BAND)
    finally:
        S.sv_free(h)
