"""Plans of default shape across the widths where their register count and tile
change (interpreted passes with half the registers, permutations folded into
write-back addresses, passes that start early), compiled passes whose gate data
is a kernel parameter, and complex128 tables applied without their cosines,
against the oracle: generic angles and the special ones where a deferred cosine
is 1, -1, zero or tiny."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2504_03967_gb300 as S
import workloads as W
from tests import gpu_util as U

pytestmark = pytest.mark.gpu

SPECIAL = [0.0, np.pi / 2, -np.pi / 2, np.pi, -np.pi, 2 * np.pi, np.pi - 1e-4, np.pi / 2 + 1e-12, 1e-9, 3.0]


def special_circuit(n, gates, seed):
    """Rotations and phases at special angles, permutations before and after
    them, on few qubits at a time so that blocks hold many gates."""
    rng = np.random.default_rng(seed)
    items = []
    ang = lambda: float(SPECIAL[rng.integers(len(SPECIAL))] if rng.random() < 0.6 else rng.uniform(-7, 7))  # noqa: E731
    while len(items) < gates:
        qs = rng.permutation(n)[: min(n, 5)]
        for _ in range(12):
            a, b = (int(q) for q in rng.permutation(qs)[:2])
            t = int(rng.choice([W.RY, W.RY, W.RX, W.RZ, W.P, W.P, W.U3, W.H, W.X, W.Z, W.CX, W.CX, W.CX, W.SWAP, W.CP, W.CZ]))
            if W.ARITY[t] == 2:
                items.append((t, (a, b), (ang(),) if t == W.CP else ()))
            else:
                items.append((t, (a,), tuple(ang() for _ in range(W.NPARAMS.get(t, 0)))))
    return W.gates_from_list(items[:gates])


def circuits(n, seed):
    rng = np.random.default_rng(seed)
    yield "special", special_circuit(n, 90, seed)
    yield "random", W.random_u3_cx(n, 3, seed)
    yield "ansatz", W.hea(n, 2, rng.uniform(0, 2 * np.pi, size=(2, n, 2)))
    yield "cx blocks", W.random_cx_blocks(n, 3 * n, seed)
    yield "qft", W.qft(n)


@pytest.mark.parametrize("dtype,n", [(S.C64, n) for n in (7, 10, 11, 12, 15, 16, 17, 18, 20, 21)] +
                         [(S.C128, n) for n in (6, 9, 10, 11, 15, 16, 18, 19)])
def test_default_plans_vs_oracle(dtype, n):
    psi0 = W.random_state(n, 3)
    for what, g in circuits(n, 10 * n + dtype):
        got = U.run_gpu(n, g, dtype, psi0=psi0)
        U.assert_close(got, U.run_oracle(n, g, psi0), dtype, "%s n=%d" % (what, n))


@pytest.mark.parametrize("dtype,n", [(S.C64, 15), (S.C128, 14)])
def test_compiled_plans_vs_oracle(dtype, n):
    psi0 = W.random_state(n, 4)
    for what, g in circuits(n, 7):
        got = U.run_gpu(n, g, dtype, psi0=psi0, jit=1)
        U.assert_close(got, U.run_oracle(n, g, psi0), dtype, "%s n=%d" % (what, n))


def test_new_angles_reuse_compiled_passes():
    """Circuits of one shape share their compiled passes whatever the angles."""
    n = 14
    rng = np.random.default_rng(5)
    g = W.random_u3_cx(n, 3, 6)
    u3 = g["type"] == W.U3
    U.run_gpu(n, g, S.C64, jit=1)
    before = S.sv_jit_stats()["compiled"]
    for _ in range(3):
        g["p"][u3] = rng.uniform(0.1, 2 * np.pi - 0.1, size=(int(u3.sum()), 3))
        near_pi = np.abs(g["p"][:, 0] - np.pi) < 0.02  # (rotations kept as general real gates)
        g["p"][near_pi & u3, 0] += 0.1
        got = U.run_gpu(n, g, S.C64, jit=1)
        U.assert_close(got, U.run_oracle(n, g), S.C64, "new angles")
    assert S.sv_jit_stats()["compiled"] == before


def test_many_deferred_factors():
    """More rotations in one pass than the deferred factors' range holds, on a
    state far from unit norm."""
    n = 10
    rng = np.random.default_rng(8)
    items = []
    for _ in range(60):
        for q in range(n):
            items.append((W.RY, (q,), (float(np.pi + rng.uniform(-0.3, 0.3)),)))
        items += [(W.CX, (q, (q + 1) % n), ()) for q in range(0, n - 1, 2)]
    g = W.gates_from_list(items)
    psi0 = W.random_state(n, 9)
    for dtype in (S.C64, S.C128):
        for opts in ({}, {"jit": 1}):
            got = U.run_gpu(n, g, dtype, psi0=1e6 * psi0, **opts) / 1e6
            U.assert_close(got, U.run_oracle(n, g, psi0), dtype, "many rotations %s" % opts)
