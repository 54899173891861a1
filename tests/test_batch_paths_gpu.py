"""sv_batch_run's circuits that leave the waves (tile widths the wave kernel does
not take, relabelling): compiled passes when asked for, memory given back."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import oracle
import paper_2504_03967_gb300 as S
import workloads as W

pytestmark = pytest.mark.gpu


def batch_run(circuits, dtype, shots, seed, **opts):
    """sv_batch_run with any option of sv_options: (samples, <Z>)."""
    ns = np.array([n for n, _ in circuits], np.int32)
    counts = np.array([len(g) for _, g in circuits], np.int64)
    offs = (np.cumsum(counts) - counts).astype(np.int64)
    gates = np.ascontiguousarray(np.concatenate([g for _, g in circuits]))
    samp = np.empty((len(circuits), shots), np.uint64)
    ez = np.empty((len(circuits), int(ns.max())))
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    o = S._opts(**opts)
    S._check(S.lib().sv_batch_run(
        ctypes.c_int(len(circuits)), p(ns), p(offs), p(counts), p(gates), ctypes.c_int(dtype), ctypes.c_uint64(shots),
        ctypes.c_uint64(seed), ctypes.byref(o), p(samp) if shots else None, p(ez), ctypes.c_int(ez.shape[1]), None))
    return samp, ez


@pytest.mark.parametrize("dtype,tile_m", [(S.C64, 12), (S.C128, 11)], ids=["c64", "c128"])
def test_batch_compiles_passes_outside_the_waves(dtype, tile_m):
    """Every pass of these plans runs compiled with jit = 1, those that end in
    CX and SWAP gates included."""
    circuits = []
    for c in range(3):
        items = [(W.RY, (q,), (0.1 + 0.2 * q + c,)) for q in range(15)]
        items += [(W.CX, (q, (q + 1) % 15), ()) for q in range(15)] + [(W.SWAP, (q, 14 - q), ()) for q in range(7)]
        circuits.append((15, W.gates_from_list(items)))
    passes = sum(S.sv_plan_circuit(n, dtype, g, tile_m=tile_m)["passes"] for n, g in circuits)
    before = S.sv_jit_stats()
    _, ez = batch_run(circuits, dtype, 0, 0, tile_m=tile_m, jit=1)
    after = S.sv_jit_stats()
    assert after["failed"] == before["failed"]
    assert after["launched"] - before["launched"] == passes
    tol = 1e-5 if dtype == S.C64 else 1e-12
    for c, (n, g) in enumerate(circuits):
        assert np.abs(ez[c, :n] - oracle.expect_z(oracle.apply_circuit(n, g))).max() <= tol


def test_batch_gives_back_the_read_out_scratch():
    """Relabelled circuits (outside the waves, read out through a logical-order
    CDF, about 1 MB of it per call): repeated calls hold no more device memory."""
    torch = pytest.importorskip("torch")
    n = 20
    g = W.gates_from_list([(W.H, (q,), ()) for q in range(n)] + [(W.SWAP, (0, n - 1), ()), (W.CX, (1, 2), ())])
    circuits = [(n, g)] * 4

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    for _ in range(3):
        batch_run(circuits, S.C64, 40000, 1, relabel=1)
    f0 = free()
    for _ in range(100):
        samp, ez = batch_run(circuits, S.C64, 40000, 1, relabel=1)
    assert f0 - free() < 32 << 20
    assert np.abs(ez).max() <= 1e-5 and samp.max() < 1 << n
