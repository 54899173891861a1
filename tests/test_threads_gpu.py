"""Handles on several host threads: the first launches of every pass kernel,
with different amounts of shared memory, at the same moment."""
from __future__ import annotations

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import threading
import numpy as np
import paper_2504_03967_gb300 as S
import workloads as W

n, threads = 15, 4
circuits = [W.random_u3_cx(n, 1 + 3 * t, t) for t in range(threads)]
kinds = [(dt, dict(tile_m=m, pass_kernel=pk, jit=-1)) for dt, ms in ((S.C64, (11, 12, 13, 14)), (S.C128, (10, 11, 12, 13)))
         for m in ms for pk in (0, 1, 2)] + [(S.C64, dict(jit=-1)), (S.C128, dict(jit=-1))]
gate = threading.Barrier(threads)
failed = []


def work(t):
    hs = {dt: S.sv_alloc(n, dt) for dt in (S.C64, S.C128)}
    for dt, opts in kinds:
        h = hs[dt]
        S.sv_init_basis(h, 0)
        S.sv_norm(h)
        gate.wait()
        try:
            S.sv_apply_circuit(h, circuits[t], **opts)
            if abs(S.sv_norm(h) - 1.0) > 1e-4:
                failed.append((dt, opts, "norm"))
        except S.SVError as e:
            failed.append((dt, opts, str(e)))
            S.sv_free(h)
            hs[dt] = S.sv_alloc(n, dt)


ts = [threading.Thread(target=work, args=(t,)) for t in range(threads)]
[t.start() for t in ts]
[t.join() for t in ts]
assert not failed, failed
"""


def test_first_launches_on_several_threads():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-2000:]
