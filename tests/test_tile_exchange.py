"""The planner's tile exchange (CPU): plans over several narrow tiles, with
multiplexors among the gates left for later, reproduce the circuit, and an
exchange never makes a plan longer than the front of the list would."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2504_03967_gb300 as S
import workloads as W
from paper_2504_03967_gb300 import build as B
from tests.oracle_pins import random_mixed_circuit
from tests.test_plan_ops import _apply_ops


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()


@pytest.mark.parametrize("tile_m", [6, 7, 8])
@pytest.mark.parametrize("seed", [4, 5])
def test_exchanges_beside_multiplexors(seed, tile_m):
    from tests.test_mux_gpu import _ladder_mix

    n = 10
    g = np.concatenate([random_mixed_circuit(n, 60, np.random.default_rng(seed)), _ladder_mix(seed),
                        W.random_u3_cx(n, 3, seed)])
    ops = S.sv_plan_ops(n, S.C64, g, mux=1, tile_m=tile_m)
    kinds = [op["kind"] for op in ops]
    assert "mux" in kinds and max(op["pass"] for op in ops) >= 4
    rng = np.random.default_rng(seed)
    psi0 = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi0 /= np.linalg.norm(psi0)
    assert np.abs(_apply_ops(n, ops, psi0) - oracle.apply_circuit(n, g, psi0)).max() < 1e-12


def test_random_circuits_need_fewer_passes():
    """8 layers on 20 qubits in 13-qubit tiles: nine passes without exchanges."""
    assert S.sv_plan_circuit(20, S.C64, W.random_u3_cx(20, 8, 1), k_max=5, tile_m=13)["passes"] <= 6
