"""The default plan of small states (half the registers, narrower tiles) as the
calls that compare, report and time plans see it."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2504_03967_gb300 as S
import workloads as W
from tests import gpu_util as U
from tests.test_small_plans_gpu import circuits

pytestmark = pytest.mark.gpu

SIZES = [(S.C64, 9), (S.C64, 13), (S.C64, 16), (S.C64, 19), (S.C64, 21), (S.C128, 9), (S.C128, 12), (S.C128, 16),
         (S.C128, 18), (S.C128, 20)]


def widths(h, g, **opts):
    S.sv_init_basis(h, 0)
    S.sv_apply_circuit(h, g, **opts)
    p = S.sv_last_plan(h)
    return p["k_max"], p["tile_m"]


@pytest.mark.parametrize("dtype,n", SIZES)
def test_cost_model_planner_is_judged_against_the_default_plan(dtype, n):
    """Without a model SV_PLAN_MLP runs the default plan; with one the judge's
    last trial of every round is the default plan."""
    g = W.random_u3_cx(n, 3, 7)
    S.sv_cost_model_unload()
    h, h2 = S.sv_alloc(n, dtype), S.sv_alloc(n, dtype)
    try:
        default = widths(h, g)
        assert widths(h, g, planner=S.PLAN_MLP) == default
        rng = np.random.default_rng(1)
        X = rng.uniform(0, 1, size=(64, S.sv_feature_count())).astype(np.float32)
        S.sv_cost_model_train(X, np.exp(X[:, 0]), epochs=50, lr=3e-3, seed=1)
        seen = [widths(h2, g, planner=S.PLAN_MLP)]
        T = len(S.sv_cost_model_last_trials(16)["predicted_ms"])
        seen += [widths(h2, g, planner=S.PLAN_MLP) for _ in range(2 * T - 1)]
        assert T > 1 and seen[T - 1] == seen[2 * T - 1] == default
    finally:
        S.sv_cost_model_unload()
        S.sv_free(h)
        S.sv_free(h2)


@pytest.mark.parametrize("dtype,n,k,m", [(S.C64, 16, 5, 13), (S.C128, 14, 4, 12)])
def test_recorded_features_tell_the_register_counts_apart(dtype, n, k, m):
    g = W.random_u3_cx(n, 3, 8)
    h = S.sv_alloc(n, dtype)
    try:
        kernel = []
        for opts in ({}, dict(k_max=k, tile_m=m), dict(k_max=k, tile_m=m, pass_kernel=1)):
            S.sv_init_basis(h, 0)
            S.sv_apply_circuit(h, g, record=1, **opts)
            kernel.append(set(S.sv_pass_times(h, features=True)[1][:, 29].tolist()))
        assert kernel == [{0.5}, {1.0}, {0.0}]
    finally:
        S.sv_free(h)


@pytest.mark.parametrize("dtype,n", [(S.C64, n) for n in range(2, 11)] + [(S.C128, n) for n in (*range(2, 10), 16, 17)])
def test_smallest_default_plans_vs_oracle(dtype, n):
    psi0 = W.random_state(n, 5)
    for what, g in circuits(n, 3 * n + dtype):
        U.assert_close(U.run_gpu(n, g, dtype, psi0=psi0), U.run_oracle(n, g, psi0), dtype, "%s n=%d" % (what, n))


def test_default_plan_shapes():
    """Block and tile width on both sides of each line of the rule."""
    want = {(S.C64, 5): (5, 5), (S.C64, 6): (3, 6), (S.C64, 9): (3, 9), (S.C64, 10): (4, 10), (S.C64, 20): (4, 12),
            (S.C64, 21): (5, 13), (S.C128, 8): (2, 8), (S.C128, 9): (3, 9), (S.C128, 16): (3, 10), (S.C128, 17): (3, 10),
            (S.C128, 18): (3, 11), (S.C128, 19): (4, 12)}
    for (dtype, n), shape in want.items():
        h = S.sv_alloc(n, dtype)
        try:
            assert widths(h, W.random_u3_cx(n, 2, 1)) == shape, (dtype, n)
        finally:
            S.sv_free(h)


@pytest.mark.parametrize("dtype,n", SIZES + [(S.C64, 14), (S.C128, 10)])
def test_reported_options_name_the_plan_that_ran(dtype, n):
    """sv_last_plan's options, handed back, give the default plan again: the
    same passes (recorded features) and, bit for bit, the same state."""
    g = W.random_u3_cx(n, 3, 9)
    runs = []
    opts = {}
    for _ in range(2):
        h = S.sv_alloc(n, dtype)
        try:
            S.sv_load_state(h, W.random_state(n, 2))
            S.sv_apply_circuit(h, g, record=1, **opts)
            p = S.sv_last_plan(h)
            opts = {k: p[k] for k in ("k_max", "tile_m", "tensor", "pass_kernel")}
            runs.append((opts, S.sv_pass_times(h, features=True)[1], S.sv_store_state(h)))
        finally:
            S.sv_free(h)
    (o1, f1, s1), (o2, f2, s2) = runs
    assert o1 == o2 and np.array_equal(f1, f2) and np.array_equal(s1, s2)


@pytest.mark.parametrize("dtype,n", [(S.C64, 8), (S.C64, 14), (S.C64, 17), (S.C128, 8), (S.C128, 14), (S.C128, 17)])
def test_autotune_times_the_default_plan(dtype, n):
    """The tuned options are no slower than passing none (best of several
    calls of each, within their noise)."""
    torch = pytest.importorskip("torch")
    g = W.random_u3_cx(n, 6, 3)
    h = S.sv_alloc(n, dtype)
    try:
        tuned, _ = S.sv_autotune(h, g)
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        best = []
        for opts in ({}, tuned):
            t = []
            for _ in range(12):
                S.sv_init_basis(h, 0)
                S.sv_norm(h)
                torch.cuda.synchronize()
                e0.record()
                S.sv_apply_circuit(h, g, **opts)
                e1.record()
                e1.synchronize()
                t.append(e0.elapsed_time(e1))
            best.append(min(t[2:]))
        assert best[1] <= 1.15 * best[0] + 0.003, (tuned, best)
    finally:
        S.sv_free(h)


@pytest.mark.parametrize("opts", [{}, dict(k_max=5, tile_m=13), dict(jit=1)], ids=["default", "wide", "compiled"])
def test_rotations_keep_the_norm(opts):
    """Rotations whose tangent 2 + 0.45 ulp rounds down: with their factor taken
    from the unrounded cosine each would lose 2 s^2 * 0.45 * 2^-23 of the norm
    squared, all with one sign.  The rest (the pass's factor rounded once per
    call, rounding of either sign) is below a quarter of that."""
    n, calls = 11, 30
    t = 2.0 + 0.45 * 2.0 ** -22
    items = [(W.RY, (q,), (2.0 * np.arctan(t),)) for q in range(n)] + [(W.CX, (q, (q + 1) % n), ()) for q in range(n)]
    g = W.gates_from_list(items)
    h = S.sv_alloc(n, S.C64)
    try:
        S.sv_load_state(h, W.random_state(n, 1))
        norm0 = S.sv_norm(h)
        for _ in range(calls):
            S.sv_apply_circuit(h, g, **opts)
        drift = 2 * 0.8 * 0.45 * 2.0 ** -23 * n * calls
        assert abs(S.sv_norm(h) ** 2 / norm0 ** 2 - 1.0) < 0.25 * drift
    finally:
        S.sv_free(h)


def test_many_passes_round_their_factor_once():
    """A 12-qubit ansatz takes 12 small passes or one wide one; with a rounding
    of every amplitude at each pass's factor (2^-24 / sqrt(3) rms, eleven of them
    more, on an error of about 3.4e-7) the mean error would be 5% larger or
    more."""
    n, layers = 12, 8
    err = {"small": [], "wide": []}
    for seed in range(6):
        g = W.hea(n, layers, np.random.default_rng(seed).uniform(0, 2 * np.pi, size=(layers, n, 2)))
        ref = U.run_oracle(n, g)
        for what, opts in (("small", {}), ("wide", dict(k_max=5, tile_m=13))):
            err[what].append(np.linalg.norm(U.run_gpu(n, g, S.C64, **opts) - ref))
    assert np.mean(err["small"]) <= 1.04 * np.mean(err["wide"])


def test_new_angles_reuse_compiled_hadamard_passes():
    """A pass that holds Hadamards only (the second of these plans) keeps its
    compiled code when the angles of the one before it change."""
    n = 14
    before = None
    for seed in range(3):
        a = np.random.default_rng(seed).uniform(0.2, 2.8, size=(2, 13))
        items = [(W.RY, (q,), (float(a[0, q]),)) for q in range(13)] + [(W.CX, (q, (q + 1) % 13), ()) for q in range(13)]
        items += [(W.RY, (q,), (float(a[1, q]),)) for q in range(13)]
        items += [(W.H, (13,), ()), (W.CX, (13, 0), ()), (W.H, (0,), ()), (W.CX, (0, 13), ()), (W.H, (13,), ())]
        g = W.gates_from_list(items)
        second = [op for op in S.sv_plan_ops(n, S.C64, g, k_max=5, tile_m=13) if op["pass"] == 1]
        assert [list(op["qubits"]) for op in second] == [[0, 13]]
        U.assert_close(U.run_gpu(n, g, S.C64, jit=1), U.run_oracle(n, g), S.C64, "seed %d" % seed)
        if seed:
            assert S.sv_jit_stats()["compiled"] == before
        before = S.sv_jit_stats()["compiled"]
