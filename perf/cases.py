"""The work this simulator is used for, as cases that can be timed.

Every case goes through the calls a user's program makes (the C ABI names of
``paper_2504_03967_gb300``).  A case is a dict of plain values:

  kind "random"   layers of U3 on every qubit and CX on a random disjoint
                  pairing, applied to a basis state; the circuit is the case's
                  (a program that runs one circuit on many inputs), the basis
                  state comes from the seed
  kind "hea"      one evaluation of a hardware-efficient ansatz (RY, RZ, CX
                  ring) from |0...0>, new angles for every seed
  kind "qft"      the QFT with its final swaps: from a basis state with the
                  swaps as a relabelling (complex64), or on a Gaussian state in
                  place
  kind "qcrank"   one QCrank image circuit from |0...0>: 2^a addresses, d data
                  qubits, 2 d 2^a + a gates
  kind "batch"    sv_batch_run over many circuits: a parameter sweep of one
                  ansatz ("hea") or small circuits of uneven size ("small")
  kind "measure"  shots and <Z_i> from one read of a given state
  kind "image"    the QCrank read-out of a given state: 3000 shots per address
                  and their decoding

Sizes are those of the repository's workloads and benchmark (12-qubit double
precision circuit, QFT on 28 qubits, QCrank with 2^14 addresses and 6 data
qubits, 20-qubit ansatz of 8 layers, random circuits up to 30 qubits with as
many layers as keep a pass well below a second).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2504_03967_gb300 as S

H, RY, RZ, U3, CX, CP, SWAP = 0, 5, 6, 8, 9, 11, 12  # gate codes of the record format
SHOTS_PER_ADDRESS = 3000


def listed():
    return [
        # a single small double-precision circuit, as in an interactive session: latency
        dict(name="random c128 n12", kind="random", dtype="c128", n=12, layers=20, circuit=1001, jit=0),
        # an ordinary medium circuit of odd width that fits the L2 cache
        dict(name="random c64 n17", kind="random", dtype="c64", n=17, layers=20, circuit=1017, jit=0),
        # one energy evaluation of a variational loop
        dict(name="hea c64 n20", kind="hea", dtype="c64", n=20, layers=8),
        # the large single-precision circuit family the benchmark runs (largest)
        dict(name="random c64 n30", kind="random", dtype="c64", n=30, layers=8, circuit=1004, jit=1),
        # the same family in double precision
        dict(name="random c128 n25", kind="random", dtype="c128", n=25, layers=3, circuit=1025, jit=1),
        # the benchmark's QFT: a basis state, swaps as a relabelling
        dict(name="qft c64 n28", kind="qft", dtype="c64", n=28, relabel=True),
        # a QFT inside a larger program: a general double-precision state, in place
        dict(name="qft c128 n24", kind="qft", dtype="c128", n=24, relabel=False),
        # one image encoded (the paper's 2^14 x 6 row)
        dict(name="qcrank c64 a14 d6", kind="qcrank", dtype="c64", a=14, d=6),
        # a parameter sweep of one ansatz
        dict(name="batch hea c64", kind="batch", of="hea", n=20, layers=8, count=256),
        # many small circuits of uneven size (the paper's parallel mode)
        dict(name="batch small c64", kind="batch", of="small", n=13, layers=6, count=1024),
        # the read-out that ends a large run: 10^5 shots and <Z_i>
        dict(name="measure c64 n28", kind="measure", dtype="c64", n=28, shots=100000),
        # the image read back: 3000 shots per address, decoded on the device
        dict(name="image c64 a14 d6", kind="image", dtype="c64", a=14, d=6),
    ]


def draw(rng):
    kind = rng.choice(["random", "random", "hea", "qft", "qcrank", "batch", "batch", "measure", "measure", "image"])
    dtype = rng.choice(["c64", "c64", "c64", "c128"])
    c64 = dtype == "c64"
    if kind == "random":
        n = rng.randint(10, 29 if c64 else 24)
        top = 20 if n < 20 else (8 if n < 26 else 4)
        return dict(kind=kind, dtype=dtype, n=n, layers=rng.randint(2, top if c64 else min(top, 40 - n)),
                    circuit=rng.randrange(1 << 20), jit=0 if n < 22 else 1)
    if kind == "hea":
        return dict(kind=kind, dtype=dtype, n=rng.randint(12, 21 if c64 else 18), layers=rng.randint(2, 10))
    if kind == "qft":
        return dict(kind=kind, dtype=dtype, n=rng.randint(12, 28 if c64 else 25), relabel=c64 and rng.random() < 0.5)
    if kind == "qcrank":
        return dict(kind=kind, dtype=dtype, a=rng.randint(7, 14), d=rng.randint(2, 8))
    if kind == "batch":
        if rng.random() < 0.5:
            n = rng.randint(14, 20)
            return dict(kind=kind, of="hea", n=n, layers=rng.randint(2, 8), count=min(256, int(2 ** rng.uniform(3, 29 - n))))
        return dict(kind=kind, of="small", n=rng.randint(9, 13), layers=rng.randint(2, 8), count=int(2 ** rng.uniform(4, 10)))
    if kind == "measure":
        return dict(kind=kind, dtype=dtype, n=rng.randint(12, 28 if c64 else 27), shots=int(10 ** rng.uniform(2, 6)))
    return dict(kind=kind, dtype="c64", a=rng.randint(6, 14), d=rng.randint(2, 7))


# ---- gate lists --------------------------------------------------------------
def _records(types, q0, q1=None, p0=None, p1=None, p2=None):
    g = np.zeros(len(types), dtype=S.GATE_DTYPE)
    g["type"] = types
    g["nq"] = np.where(np.isin(g["type"], (CX, CP, SWAP)), 2, 1)
    g["q"][:, 0] = q0
    if q1 is not None:
        g["q"][:, 1] = q1
    for i, p in enumerate((p0, p1, p2)):
        if p is not None:
            g["p"][:, i] = p
    return g


def _random_gates(n, layers, seed):
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(layers):
        ang = rng.uniform(0.0, 2.0 * np.pi, size=(n, 3))
        out.append(_records(np.full(n, U3), np.arange(n), None, ang[:, 0], ang[:, 1], ang[:, 2]))
        pairs = rng.permutation(n)[: n // 2 * 2].reshape(-1, 2)
        out.append(_records(np.full(len(pairs), CX), pairs[:, 0], pairs[:, 1]))
    return np.concatenate(out)


def _hea_gates(n, layers, angles):
    q = np.arange(n)
    out = []
    for l in range(layers):
        rot = _records(np.tile([RY, RZ], n), np.repeat(q, 2), None, angles[l].reshape(-1))
        out += [rot, _records(np.full(n, CX), q, (q + 1) % n)]
    return np.concatenate(out)


def _qft_gates(n):
    out = []
    for j in range(n - 1, -1, -1):
        out.append(_records([H], [j]))
        k = np.arange(j - 1, -1, -1)
        if len(k):
            out.append(_records(np.full(j, CP), k, j, np.pi * np.ldexp(1.0, -(j - k))))
    i = np.arange(n // 2)
    out.append(_records(np.full(len(i), SWAP), i, n - 1 - i))
    return np.concatenate(out)


def _qcrank_gates(a, d, pixels):
    """H on the address qubits, then per data qubit a ladder of RY and CX along
    the Gray code whose angles are the Walsh-Hadamard transform of the pixels'."""
    L = 1 << a
    w = np.pi * pixels
    h = 1
    while h < L:
        w = w.reshape(L // (2 * h), 2, h, d)
        w = np.stack([w[:, 0] + w[:, 1], w[:, 0] - w[:, 1]], axis=1).reshape(L, d)
        h *= 2
    i = np.arange(L)
    gray = i ^ (i >> 1)
    flips = gray ^ np.roll(gray, -1)
    ctrl = np.log2(flips).astype(np.int64)
    lad = np.zeros((d, L, 2), dtype=S.GATE_DTYPE)
    t = (a + np.arange(d))[:, None]
    lad["type"][:, :, 0], lad["type"][:, :, 1] = RY, CX
    lad["nq"][:, :, 0], lad["nq"][:, :, 1] = 1, 2
    lad["q"][:, :, 0, 0], lad["q"][:, :, 1, 0], lad["q"][:, :, 1, 1] = t, ctrl[None, :], t
    lad["p"][:, :, 0, 0] = (w[gray] / L).T
    return np.concatenate([_records(np.full(a, H), np.arange(a)), lad.reshape(-1)])


def _pixels(case, seed):
    return np.random.default_rng(seed).uniform(0.0, 1.0, size=(1 << case["a"], case["d"]))


def _batch(case, seed):
    """[(n, gates), ...] of a batch case."""
    rng = np.random.default_rng(seed)
    n, layers, count = case["n"], case["layers"], case["count"]
    if case["of"] == "hea":
        return [(n, _hea_gates(n, layers, rng.uniform(0.0, 2.0 * np.pi, size=(layers, n, 2)))) for _ in range(count)]
    sizes = rng.integers(6, n + 1, size=count)
    sizes[0] = n
    return [(int(m), _random_gates(int(m), layers, int(rng.integers(1 << 30)))) for m in sizes]


# ---- states --------------------------------------------------------------------
class _Handle:
    """A state's device memory and the library's handle on it."""

    def __init__(self, n, dtype, amps=None):
        self.amps = amps if amps is not None else torch.zeros(
            1 << n, dtype=torch.complex64 if dtype == "c64" else torch.complex128, device="cuda")
        self.h = S.sv_attach(n, S.C64 if dtype == "c64" else S.C128, self.amps.data_ptr(),
                             torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        if getattr(self, "h", None):
            S.sv_free(self.h)
            self.h = None


def _gaussian(n, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    v = torch.randn((1 << n, 2), generator=g, device="cuda", dtype=torch.float32)
    v = torch.view_as_complex(v if dtype == "c64" else v.double())
    return v.div_(torch.linalg.vector_norm(v))


def _qcrank_state(a, d, pixels):
    """The state a QCrank circuit prepares, in 64 bits: amplitude of address j
    and data bits b is 2^(-a/2) times cos or sin of half of pi * pixel per bit."""
    th = torch.from_numpy(0.5 * np.pi * pixels).cuda()
    psi = torch.full((1, 1 << a), 2.0 ** (-0.5 * a), dtype=torch.float64, device="cuda")
    for k in range(d):
        psi = torch.cat([psi * torch.cos(th[:, k]), psi * torch.sin(th[:, k])])
    return psi.reshape(-1)


def _basis(case, seed):
    return int(np.random.default_rng(seed).integers(0, 1 << case["n"]))


def prepare(case, seed):
    kind, st = case["kind"], dict(case=case, seed=seed)
    if kind == "random":
        st.update(state=_Handle(case["n"], case["dtype"]), gates=_random_gates(case["n"], case["layers"], case["circuit"]),
                  x=_basis(case, seed), options=dict(jit=case["jit"]))
    elif kind == "hea":
        ang = np.random.default_rng(seed).uniform(0.0, 2.0 * np.pi, size=(case["layers"], case["n"], 2))
        st.update(state=_Handle(case["n"], case["dtype"]), gates=_hea_gates(case["n"], case["layers"], ang), x=0, options={})
    elif kind == "qft":
        if case["relabel"]:
            st.update(state=_Handle(case["n"], case["dtype"]), x=_basis(case, seed), options=dict(relabel=1, jit=1))
        else:
            st.update(state=_Handle(case["n"], case["dtype"], _gaussian(case["n"], case["dtype"], seed)), x=None, options={})
        st["gates"] = _qft_gates(case["n"])
    elif kind == "qcrank":
        st.update(state=_Handle(case["a"] + case["d"], case["dtype"]),
                  gates=_qcrank_gates(case["a"], case["d"], _pixels(case, seed)), x=0, options={})
    elif kind == "batch":
        circuits = _batch(case, seed)
        sizes = np.array([n for n, _ in circuits])
        st.update(circuits=circuits, written=np.arange(sizes.max())[None, :] < sizes[:, None])
    elif kind == "measure":
        st.update(state=_Handle(case["n"], case["dtype"], _gaussian(case["n"], case["dtype"], seed)),
                  samples=torch.empty(case["shots"], dtype=torch.int64, device="cuda"),
                  expz=torch.empty(case["n"], dtype=torch.float64, device="cuda"))
    else:
        a, d = case["a"], case["d"]
        amps = _qcrank_state(a, d, _pixels(case, seed)).to(torch.complex64)
        st.update(state=_Handle(a + d, case["dtype"], amps),
                  samples=torch.empty(SHOTS_PER_ADDRESS << a, dtype=torch.int64, device="cuda"),
                  counts=torch.empty(1 << a, dtype=torch.int64, device="cuda"),
                  ones=torch.empty((1 << a, d), dtype=torch.int64, device="cuda"),
                  pixels=torch.empty((1 << a, d), dtype=torch.float64, device="cuda"))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        # <Z_i> of a single-precision simulation, kept in single precision
        _, ez = S.sv_batch_run(st["circuits"], dtype=S.C64)
        return np.where(st["written"], ez, 0.0).astype(np.float32)
    hd = st["state"]
    if kind == "measure":
        S.sv_measure_device(hd.h, case["shots"], st["seed"], st["samples"].data_ptr(), st["expz"].data_ptr())
        return [st["samples"], st["expz"]]
    if kind == "image":
        S.sv_sample_device(hd.h, len(st["samples"]), st["seed"], st["samples"].data_ptr())
        S.sv_qcrank_decode_device(st["samples"].data_ptr(), len(st["samples"]), case["a"], case["d"], st["counts"].data_ptr(),
                                  st["ones"].data_ptr(), st["pixels"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return [st["samples"], st["counts"], st["ones"], st["pixels"]]
    if st["x"] is not None:
        S.sv_init_basis(hd.h, st["x"])
    S.sv_apply_circuit(hd.h, st["gates"], **st["options"])
    return hd.amps


# ---- what a pass cannot do without ------------------------------------------------
# floating-point operations per amplitude of one gate: U3 a complex 2x2, RY a
# real 2x2, RZ a phase, H a butterfly, CP a phase on a quarter; CX and SWAP move
def work(case):
    kind = case["kind"]
    if kind == "batch":
        if case["of"] == "hea":
            amps = float(case["count"]) * 2.0 ** case["n"]
            return dict(bytes=8.0 * case["count"] * case["n"], flops=amps * case["layers"] * case["n"] * 12.0)
        per = [(m, 2.0 ** m * m * case["layers"] * 14.0) for m in range(6, case["n"] + 1)]
        return dict(bytes=8.0 * case["count"] * case["n"], flops=case["count"] * sum(f for _, f in per) / len(per))
    if kind == "image":
        a, d, shots = case["a"], case["d"], float(SHOTS_PER_ADDRESS << case["a"])
        return dict(bytes=8.0 * 2 ** (a + d) + 8.0 * shots + 8.0 * 2 ** a * (1 + 2 * d), flops=3.0 * 2 ** (a + d))
    n = case["a"] + case["d"] if kind == "qcrank" else case["n"]
    N, amp = 2.0 ** n, 8.0 if case["dtype"] == "c64" else 16.0
    if kind == "measure":
        return dict(bytes=amp * N + 8.0 * (case["shots"] + n), flops=3.0 * N)
    if kind == "random":
        return dict(bytes=amp * N, flops=14.0 * N * n * case["layers"])
    if kind == "hea":
        return dict(bytes=amp * N, flops=12.0 * N * n * case["layers"])
    if kind == "qft":
        return dict(bytes=amp * N * (1 if case["relabel"] else 2), flops=N * (4.0 * n + 1.5 * n * (n - 1) / 2))
    return dict(bytes=amp * N + 96.0 * case["d"] * 2 ** case["a"], flops=N * 6.0 * case["d"])


# ---- 64-bit values ------------------------------------------------------------------
def _u3(t, f, l):
    c, s = math.cos(0.5 * t), math.sin(0.5 * t)
    e = lambda x: complex(math.cos(x), math.sin(x))  # noqa: E731
    return c, -e(l) * s, e(f) * s, e(f + l) * c


def _apply_2x2(psi, q, m):
    v = psi.view(-1, 2, 1 << q)
    a, b = v[:, 0].clone(), v[:, 1]
    v[:, 0].mul_(m[0]).add_(b, alpha=m[1])
    b.mul_(m[3]).add_(a, alpha=m[2])


def _apply_cx(psi, c, t):
    lo, hi = min(c, t), max(c, t)
    v = psi.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
    one = v[:, 1] if c == hi else v[:, :, :, 1]
    x, y = (one[:, :, 0], one[:, :, 1]) if c == hi else (one[:, 0], one[:, 1])
    old = x.clone()
    x.copy_(y)
    y.copy_(old)


def _simulate(n, gates, x=0):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[x] = 1.0
    for t, q, p in zip(gates["type"].tolist(), gates["q"].tolist(), gates["p"].tolist()):
        if t == U3:
            _apply_2x2(psi, q[0], _u3(*p))
        elif t == RY:
            c, s = math.cos(0.5 * p[0]), math.sin(0.5 * p[0])
            _apply_2x2(psi, q[0], (c, -s, s, c))
        elif t == RZ:
            v = psi.view(-1, 2, 1 << q[0])
            v[:, 0].mul_(complex(math.cos(0.5 * p[0]), -math.sin(0.5 * p[0])))
            v[:, 1].mul_(complex(math.cos(0.5 * p[0]), math.sin(0.5 * p[0])))
        else:
            _apply_cx(psi, q[0], q[1])
    return psi


def _expect_z(p, n):
    return torch.stack([(v := p.view(-1, 2, 1 << q))[:, 0].sum() - v[:, 1].sum() for q in range(n)])


def _mass(psi):
    return psi.real.double().square() + psi.imag.double().square()


def _reverse_bits(x, n):
    r = torch.zeros_like(x)
    for b in range(n):
        r |= ((x >> b) & 1) << (n - 1 - b)
    return r


def _drawn_uniforms(shots, seed):
    """Word s of the Philox4x64-10 stream with key (seed, 0), counters from 0."""
    raw = np.random.Philox(key=int(seed), counter=2 ** 256 - 1).random_raw(shots)
    return torch.from_numpy((raw >> np.uint64(11)).astype(np.float64) * 2.0 ** -53).cuda()


def exact(case, seed):
    kind = case["kind"]
    if kind == "random":
        return _simulate(case["n"], _random_gates(case["n"], case["layers"], case["circuit"]), _basis(case, seed))
    if kind == "hea":
        ang = np.random.default_rng(seed).uniform(0.0, 2.0 * np.pi, size=(case["layers"], case["n"], 2))
        return _simulate(case["n"], _hea_gates(case["n"], case["layers"], ang))
    if kind == "qft":
        n = case["n"]
        if not case["relabel"]:
            psi = _gaussian(n, case["dtype"], seed).to(torch.complex128)
            return torch.fft.ifft(psi) * 2.0 ** (0.5 * n)
        # amplitude y of QFT|x> is 2^(-n/2) exp(2 pi i x y / 2^n); the swaps are
        # a relabelling, so it is stored at the reversed index
        y = _reverse_bits(torch.arange(1 << n, device="cuda"), n)
        ph = ((y * _basis(case, seed)) & ((1 << n) - 1)).double().mul_(2.0 * np.pi * 2.0 ** -n)
        return torch.polar(torch.full_like(ph, 2.0 ** (-0.5 * n)), ph)
    if kind == "qcrank":
        return torch.complex(p := _qcrank_state(case["a"], case["d"], _pixels(case, seed)), torch.zeros_like(p))
    if kind == "batch":
        circuits = _batch(case, seed)
        out = torch.zeros((len(circuits), max(n for n, _ in circuits)), dtype=torch.float64, device="cuda")
        if case["n"] > 16 and len(circuits) * case["layers"] > 4096:
            return None
        for i, (n, g) in enumerate(circuits):
            out[i, :n] = _expect_z(_mass(_simulate(n, g)), n)
        return out
    if kind == "measure":
        return [None, _expect_z(_mass(_gaussian(case["n"], case["dtype"], seed)), case["n"])]
    a, d = case["a"], case["d"]
    cdf = torch.cumsum(_mass(_qcrank_state(a, d, _pixels(case, seed)).to(torch.complex64)), 0)
    u = _drawn_uniforms(SHOTS_PER_ADDRESS << a, seed) * cdf[-1]
    x = torch.searchsorted(cdf, u, right=True).clamp_(max=len(cdf) - 1)
    j = x & ((1 << a) - 1)
    counts = torch.bincount(j, minlength=1 << a).double()
    ones = torch.stack([torch.bincount(j[((x >> (a + k)) & 1) == 1], minlength=1 << a) for k in range(d)], 1).double()
    return [None, None, None, torch.asin(torch.sqrt(ones / counts[:, None])) * (2.0 / np.pi)]
