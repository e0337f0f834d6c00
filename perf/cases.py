"""Measured cases: the work users of the simulator have it do, through its public entry points.

The circuits are the framework's own workload families (random layers, quantum volume, QFT,
hardware-efficient ansatz, noisy trajectories), written out here so that `exact` needs nothing but
torch and numpy.  A gate is (kind, qubits, params) as `make_gates` takes it."""
import cmath
import math

import numpy as np
import torch

import paper_2102_02957_gb300 as sv

TWO_PI = 2.0 * math.pi
DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # A short circuit on a small double-precision state by the plain method, as one checks a
        # circuit or compares methods: 480 gates of a few microseconds, launches and latency.
        dict(name="layers16_c128_plain", kind="circuit", circuit="layers", n=16, depth=20, dtype="c128", plain=True),
        # One evaluation of a variational ansatz: new angles, kept plan, state from |0..0>, three
        # Pauli expectation values read back (20 qubits, 10 layers, tensor-core groups).
        dict(name="ansatz20_c64", kind="ansatz", n=20, depth=10, dtype="c64", chunk=12, pinned=4, tc=True, terms=3),
        # Quantum volume at 30 qubits, the headline workload's family and options, at the depth of
        # 10 layers usual for this circuit: gathered chunks, look-ahead choice, tensor-core groups.
        dict(name="qv30_c64_tc", kind="circuit", circuit="qv", n=30, depth=10, dtype="c64", chunk=12, pinned=5, tc=True, look=True),
        # Random layers on an odd qubit count with the options a caller gets by default: contiguous
        # chunks of 13 bits, chunk_swap passes, FP32 register groups; continues from a state in hand.
        dict(name="layers27_c64_default", kind="circuit", circuit="layers", n=27, depth=10, dtype="c64", resume=True),
        # The same family in double precision with the layout of the method's paper and 12-bit chunks.
        dict(name="layers27_c128", kind="circuit", circuit="layers", n=27, depth=8, dtype="c128", chunk=12, resume=True),
        # QFT of a basis state in double precision, diagonal gates taken outside their chunks.
        dict(name="qft28_c128_diag", kind="circuit", circuit="qft", n=28, depth=1, dtype="c128", chunk=12, diag=True),
        # Dense two-qubit gates in double precision on gathered chunks.
        dict(name="qv25_c128_gather", kind="circuit", circuit="qv", n=25, depth=10, dtype="c128", chunk=12, pinned=4, look=True),
        # Noisy trajectories of uneven sizes and ansatz parameter sets in one graph-replayed launch.
        dict(name="batch_traj80", kind="batch", count=80, lo=12, hi=22, depth=30, p=1e-3, hea_n=20, hea_sets=16, hea_layers=10, chunk=13, tc=True),
        # What a run reads out at its end: norm, four Pauli words, 4096 shots, all probabilities.
        dict(name="readout28_c64", kind="readout", n=28, dtype="c64", words=4, shots=4096),
        # A state kept in pinned host memory, the device holding an eighth of it.
        dict(name="host26_c64", kind="host", circuit="layers", n=26, depth=4, dtype="c64", chunk=12, share=8),
        # Gate after gate at full size, one sweep each: the baseline the blocked path is held against.
        dict(name="qv28_c64_plain", kind="circuit", circuit="qv", n=28, depth=1, dtype="c64", plain=True, resume=True),
        # The section-time network: predictions, and the gradient of one training batch.
        dict(name="costmodel_grad4096", kind="model", rows=4096),
    ]


def draw(rng):
    """One more case of the listed ones' ranges; qubit counts are uniform (their work doubles per qubit)."""
    pick = rng.choice(["plain", "plain", "ansatz", "qv_tc", "layers64", "layers128", "layers128", "qft", "qv128", "batch", "readout", "host", "model"])
    if pick == "plain":
        n, dt = rng.randint(9, 27), rng.choice(["c64", "c128"])
        circuit = rng.choice(["layers", "qv", "hea"])
        return dict(kind="circuit", circuit=circuit, n=n, depth=max(1, rng.randint(8, 20) // (1 + max(0, n - 16))), dtype=dt, plain=True, resume=rng.random() < 0.5)
    if pick == "ansatz":
        return dict(kind="ansatz", n=rng.randint(13, 24), depth=rng.randint(4, 10), dtype=rng.choice(["c64", "c64", "c128"]), chunk=rng.choice([11, 12, 13]), pinned=4, tc=rng.random() < 0.7, terms=rng.randint(1, 5))
    if pick == "qv_tc":
        return dict(kind="circuit", circuit=rng.choice(["qv", "qv", "layers"]), n=rng.randint(18, 30), depth=rng.randint(5, 10), dtype="c64", chunk=rng.choice([12, 12, 13]), pinned=rng.choice([4, 5]), tc=True, look=rng.random() < 0.7)
    if pick == "layers64":
        return dict(kind="circuit", circuit=rng.choice(["layers", "qv", "hea"]), n=rng.randint(12, 27), depth=rng.randint(3, 10), dtype="c64", chunk=rng.choice([11, 12, 13]), pinned=rng.choice([0, 0, 4]), resume=rng.random() < 0.5)
    if pick == "layers128":
        return dict(kind="circuit", circuit=rng.choice(["layers", "layers", "hea"]), n=rng.randint(12, 27), depth=rng.randint(3, 8), dtype="c128", chunk=rng.choice([10, 11, 12]), pinned=rng.choice([0, 0, 4]), resume=rng.random() < 0.5)
    if pick == "qft":
        return dict(kind="circuit", circuit="qft", n=rng.randint(14, 28), depth=1, dtype=rng.choice(["c64", "c128"]), chunk=rng.choice([11, 12]), diag=rng.random() < 0.7)
    if pick == "qv128":
        return dict(kind="circuit", circuit="qv", n=rng.randint(13, 25), depth=rng.randint(3, 10), dtype="c128", chunk=rng.choice([11, 12]), pinned=rng.choice([0, 4]), look=rng.random() < 0.5)
    if pick == "batch":
        lo = rng.randint(7, 14)
        return dict(kind="batch", count=rng.randint(8, 80), lo=lo, hi=rng.randint(lo + 2, 21), depth=rng.randint(10, 30), p=rng.choice([1e-3, 1e-2]), hea_n=rng.randint(8, 20), hea_sets=rng.randint(1, 16), hea_layers=rng.randint(3, 10), chunk=rng.choice([11, 12, 13]), tc=rng.random() < 0.7)
    if pick == "readout":
        return dict(kind="readout", n=rng.randint(12, 27), dtype=rng.choice(["c64", "c128"]), words=rng.randint(1, 6), shots=rng.choice([100, 1000, 5000]))
    if pick == "host":
        return dict(kind="host", circuit=rng.choice(["layers", "qv"]), n=rng.randint(20, 26), depth=rng.randint(2, 4), dtype=rng.choice(["c64", "c128"]), chunk=rng.choice([11, 12]), share=rng.choice([4, 8]))
    return dict(kind="model", rows=rng.choice([1, 3]) * rng.randint(1, 3000))


# ------------------------------------------------------------------ inputs
def _rng(case, seed):
    return np.random.Generator(np.random.PCG64([int(seed) & 0xFFFFFFFF, int(case.get("n", 0))]))


def _layers(rng, n, depth):
    gates = []
    for _ in range(depth):
        ang = rng.uniform(0.0, TWO_PI, size=(n, 3)).tolist()
        gates += [("u3", (q,), tuple(ang[q])) for q in range(n)]
        perm = rng.permutation(n).tolist()
        gates += [("cx", (perm[2 * i], perm[2 * i + 1]), ()) for i in range(n // 2)]
    return gates


def _qv(rng, n, depth):
    """Per layer a random pairing and a Haar-random unitary on each pair (QR of a Ginibre matrix, phases of R moved into Q)."""
    gates = []
    for _ in range(depth):
        perm = rng.permutation(n).tolist()
        z = rng.standard_normal((n // 2, 4, 4)) + 1j * rng.standard_normal((n // 2, 4, 4))
        q, r = np.linalg.qr(z)
        d = np.diagonal(r, axis1=1, axis2=2)
        q = q * (d / np.abs(d))[:, None, :]
        gates += [("unitary", (perm[2 * i], perm[2 * i + 1]), (np.ascontiguousarray(q[i]),)) for i in range(n // 2)]
    return gates


def _qft(n):
    gates = []
    for j in range(n - 1, -1, -1):
        gates.append(("h", (j,), ()))
        gates += [("cp", (m, j), (math.pi / float(1 << (j - m)),)) for m in range(j - 1, -1, -1)]
    return gates + [("swap", (i, n - 1 - i), ()) for i in range(n // 2)]


def _hea(rng, n, depth):
    gates = []
    for _ in range(depth):
        gates += [("ry", (q,), (t,)) for q, t in enumerate(rng.uniform(0.0, TWO_PI, size=n).tolist())]
        gates += [("cz", (q, q + 1), ()) for q in range(n - 1)]
    return gates + [("ry", (q,), (t,)) for q, t in enumerate(rng.uniform(0.0, TWO_PI, size=n).tolist())]


def _noisy(rng, n, depth, p):
    """Depolarizing trajectory: after each gate, with probability p, a random non-identity Pauli word on its qubits."""
    base = _layers(rng, n, depth)
    hit = rng.random(len(base)) < p
    gates = []
    for g, h in zip(base, hit.tolist()):
        gates.append(g)
        if h:
            k = int(rng.integers(1, 4 ** len(g[1])))
            gates += [("xyz"[((k >> (2 * j)) & 3) - 1], (q,), ()) for j, q in enumerate(g[1]) if (k >> (2 * j)) & 3]
    return gates


def _circuit(case, seed):
    rng, n, d = _rng(case, seed), case["n"], case["depth"]
    c = case["circuit"]
    return _layers(rng, n, d) if c == "layers" else _qv(rng, n, d) if c == "qv" else _qft(n) if c == "qft" else _hea(rng, n, d)


def _batch_circuits(case, seed):
    rng = _rng(case, seed)
    # the sizes are the case's own, the circuits the seed's
    ns = [int(v) for v in np.random.Generator(np.random.PCG64(case["count"])).integers(case["lo"], case["hi"] + 1, size=case["count"])]
    gates = [_noisy(rng, n, case["depth"], case["p"]) for n in ns]
    for _ in range(case["hea_sets"]):
        ns.append(case["hea_n"])
        gates.append(_hea(rng, case["hea_n"], case["hea_layers"]))
    return ns, gates


def _ctype(case):
    return torch.complex128 if case["dtype"] == "c128" else torch.complex64


def _random_state(case, seed):
    """A normalised complex Gaussian state, as a deep random circuit leaves one."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + case["n"])
    v = torch.randn(2 << case["n"], dtype=torch.float64 if case["dtype"] == "c128" else torch.float32, device=DEV, generator=g)
    v /= math.sqrt(2.0 * (1 << case["n"]))
    return torch.view_as_complex(v.view(-1, 2))


def _basis(case, seed):
    return int(_rng(case, seed + 17).integers(0, 1 << case["n"])) if case.get("circuit") == "qft" else 0


def _plan_options(case):
    o = {}
    if "chunk" in case:
        o["chunk_bits"] = case["chunk"]
    if case.get("pinned"):
        o["gather_pinned"] = case["pinned"]
    if case.get("tc"):
        o["use_tc"] = 1
    if case.get("look") and case.get("pinned"):
        o["lookahead"] = 1
    if case.get("diag"):
        o["diag_outside"] = 1
    return o


def _words(case, seed, count):
    """Pauli words as (x mask, z mask): weights from one qubit to all of them."""
    rng, n, out = _rng(case, seed + 5), case["n"], []
    for k in range(count):
        on = rng.random(n) < (k + 1) / count
        w = rng.integers(1, 4, size=n)
        out.append((sum(1 << q for q in range(n) if on[q] and w[q] & 1), sum(1 << q for q in range(n) if on[q] and w[q] & 2)))
    return out


def _model_inputs(case, seed):
    """Network parameters (He-uniform weights, small biases), feature rows and standardised targets."""
    rng = _rng(case, seed)
    p = [rng.uniform(-1, 1, 64 * 16) * math.sqrt(6 / 16), rng.uniform(-0.1, 0.1, 64), rng.uniform(-1, 1, 64 * 64) * math.sqrt(6 / 64),
         rng.uniform(-0.1, 0.1, 64), rng.uniform(-1, 1, 64) * math.sqrt(6 / 64), rng.uniform(-0.1, 0.1, 1)]
    return (np.concatenate(p).astype(np.float32), rng.uniform(0, 1, (case["rows"], 16)).astype(np.float32), rng.standard_normal(case["rows"]).astype(np.float32))


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    stream = torch.cuda.current_stream()
    if kind == "model":
        p, s["x"], s["t"] = _model_inputs(case, seed)
        s["model"] = sv.CostModel(0)
        s["model"].set_params(p)
        return s
    if kind == "batch":
        ns, desc = _batch_circuits(case, seed)
        s["gates"] = [sv.make_gates(d) for d in desc]
        off = np.concatenate([[0], np.cumsum([max(1 << n, 32) for n in ns])])
        s["buffer"] = torch.zeros(int(off[-1]), dtype=torch.complex64, device=DEV)
        s["states"] = [sv.StateVector(n, dtype="c64", buffer=s["buffer"][int(off[i]):int(off[i]) + (1 << n)], stream=stream) for i, n in enumerate(ns)]
        opts = dict(chunk_bits=case["chunk"])
        if case["tc"]:
            opts["use_tc"] = 1
        s["batch"] = sv.Batch(s["states"], s["gates"], **opts)
        return s
    if kind == "host":
        s["gates"] = sv.make_gates(_circuit(case, seed))
        s["plan"] = sv.Plan(case["n"], s["gates"], **_plan_options(case))
        amps = _random_state(case, seed)
        s["host"] = torch.empty(amps.shape, dtype=amps.dtype, pin_memory=True)
        s["host"].copy_(amps)
        s["work"] = torch.empty(amps.numel() // case["share"], dtype=amps.dtype, device=DEV)
        return s
    if kind == "readout" or case.get("resume"):
        s["buffer"] = _random_state(case, seed)
    else:
        s["buffer"] = torch.zeros(1 << case["n"], dtype=_ctype(case), device=DEV)
    s["state"] = sv.StateVector(case["n"], dtype=case["dtype"], buffer=s["buffer"], stream=stream)
    if kind == "readout":
        s["words"] = _words(case, seed, case["words"])
        s["probs"] = torch.empty(1 << case["n"], dtype=torch.float64, device=DEV)
        s["seed"] = int(seed) + 99
        return s
    if kind == "ansatz":
        s["desc"] = _hea(_rng(case, seed), case["n"], case["depth"])
        s["words"] = _words(case, seed, case["terms"])
        s["plan"] = sv.Plan(case["n"], sv.make_gates(s["desc"]), **_plan_options(case))
        return s
    s["gates"] = sv.make_gates(_circuit(case, seed))
    s["plan"] = None if case.get("plain") else sv.Plan(case["n"], s["gates"], **_plan_options(case))
    s["basis"] = None if case.get("resume") else _basis(case, seed)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "model":
        y = s["model"].forward(s["x"])
        grad, loss = s["model"].gradient(s["x"], s["t"])
        return {"y": y, "grad": grad, "loss": loss}
    if kind == "batch":
        s["batch"].run(use_graph=True, from_zero=True)
        return s["buffer"]
    if kind == "host":
        sv.apply_host(case["n"], s["host"], s["gates"], s["plan"], s["work"].numel() * s["work"].element_size(), dtype=case["dtype"], dev_work=s["work"].data_ptr(),
                      stream=torch.cuda.current_stream())
        return s["host"]
    st = s["state"]
    if kind == "readout":
        return {"norm2": st.norm2(), "words": np.array([st.expval_pauli(x, z) for x, z in s["words"]]), "shots": st.sample(case["shots"], s["seed"]).astype(np.int64),
                "probs": st.probabilities(s["probs"])}
    if kind == "ansatz":
        st.init_basis(0)
        st.apply(sv.make_gates(s["desc"]), s["plan"])
        return {"state": s["buffer"], "words": np.array([st.expval_pauli(x, z) for x, z in s["words"]])}
    if s["basis"] is not None:
        st.init_basis(s["basis"])
    st.apply(s["gates"], s["plan"])
    return s["buffer"]


# ------------------------------------------------------------------ what a pass cannot do without
#: real operations per amplitude: dense 1-qubit (2 complex products and a sum), dense 2-qubit, real rotations, a phase on a quarter of the state
_FLOPS = {"u3": 14.0, "unitary": 30.0, "ry": 6.0, "h": 4.0, "cp": 1.5}


def _gate_flops(circuit, n, depth):
    per = {"layers": n * depth * _FLOPS["u3"], "qv": (n // 2) * depth * _FLOPS["unitary"], "qft": n * _FLOPS["h"] + n * (n - 1) / 2 * _FLOPS["cp"],
           "hea": n * (depth + 1) * _FLOPS["ry"]}
    return per[circuit] * float(1 << n)


def work(case):
    kind = case["kind"]
    if kind == "model":
        return {"bytes": 4.0 * (case["rows"] * 18 + 3 * 5313), "flops": 8.0 * 5313 * case["rows"]}
    if kind == "batch":
        ns = np.random.Generator(np.random.PCG64(case["count"])).integers(case["lo"], case["hi"] + 1, size=case["count"]).tolist()
        b = 8.0 * (sum(1 << n for n in ns) + case["hea_sets"] * (1 << case["hea_n"]))
        f = sum(_gate_flops("layers", n, case["depth"]) for n in ns) + case["hea_sets"] * _gate_flops("hea", case["hea_n"], case["hea_layers"])
        return {"bytes": b, "flops": f}
    amp = 16 if case["dtype"] == "c128" else 8
    size = float(amp << case["n"])
    if kind == "readout":
        return {"bytes": size + 8.0 * (1 << case["n"]), "flops": (4.0 + 8.0 * case["words"]) * (1 << case["n"])}
    # a run from a basis state writes the state; one that resumes reads it too
    both = case.get("resume") or kind == "host"
    return {"bytes": size * (2 if both else 1), "flops": _gate_flops(case.get("circuit", "hea"), case["n"], case["depth"])}


# ------------------------------------------------------------------ the same in 64 bits, by torch and numpy
def _matrix(kind, qs, ps):
    """(qubits from low to high local bit, row-major matrix)."""
    if kind == "u3":
        t, p, l = ps
        c, s = math.cos(t / 2), math.sin(t / 2)
        return qs, np.array([[c, -cmath.exp(1j * l) * s], [cmath.exp(1j * p) * s, cmath.exp(1j * (p + l)) * c]])
    if kind == "ry":
        c, s = math.cos(ps[0] / 2), math.sin(ps[0] / 2)
        return qs, np.array([[c, -s], [s, c]], dtype=complex)
    if kind == "cx":
        return (qs[1], qs[0]), np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 0, 1], [0, 0, 1, 0]], dtype=complex)
    if kind == "cz":
        return qs, np.diag([1, 1, 1, -1]).astype(complex)
    if kind in "xyz":
        return qs, {"x": np.array([[0, 1], [1, 0]], dtype=complex), "y": np.array([[0, -1j], [1j, 0]]), "z": np.diag([1, -1]).astype(complex)}[kind]
    return qs, np.asarray(ps[0])


def _apply(v, n, gate):
    """One gate on the 2^n complex128 tensor v; returns the new tensor (v itself where it can be changed in place)."""
    qs, m = _matrix(*gate)
    order = sorted(qs)
    if len(qs) == 1:
        view = lambda t: t.view(1 << (n - 1 - qs[0]), 2, 1 << qs[0])  # noqa: E731
        part = lambda t, b: t[:, b]  # noqa: E731
    else:
        lo, hi = order
        view = lambda t: t.view(1 << (n - 1 - hi), 2, 1 << (hi - lo - 1), 2, 1 << lo)  # noqa: E731
        at = {q: j for j, q in enumerate(qs)}
        part = lambda t, b: t[:, (b >> at[hi]) & 1, :, (b >> at[lo]) & 1]  # noqa: E731
    dim = len(m)
    a = view(v)
    rows = [r for r in range(dim) if not (m[r, r] == 1 and np.count_nonzero(m[r]) == 1)]
    if all(np.count_nonzero(m[r]) == 1 for r in range(dim)):  # a permutation with phases
        old = [part(a, int(np.flatnonzero(m[r])[0])).clone() for r in rows]
        for r, x in zip(rows, old):
            z = complex(m[r][np.flatnonzero(m[r])[0]])
            part(a, r).copy_(x if z == 1 else x * z)
        return v
    new = torch.empty_like(v)
    b = view(new)
    for r in range(dim):
        o = part(b, r)
        torch.mul(part(a, 0), complex(m[r, 0]), out=o)
        for c in range(1, dim):
            if m[r, c] != 0:
                o.add_(part(a, c), alpha=complex(m[r, c]))
    return new


def _simulate(v, n, gates):
    for g in gates:
        v = _apply(v, n, g)
    return v


def _zero(n):
    v = torch.zeros(1 << n, dtype=torch.complex128, device=DEV)
    v[0] = 1
    return v


def _expval(v, n, x, z):
    j = torch.arange(1 << n, device=DEV, dtype=torch.int64)
    u = v[j ^ x].conj() * v
    par = j & z
    for sh in (32, 16, 8, 4, 2, 1):
        par = par ^ (par >> sh)
    r = complex((u * (1 - 2 * (par & 1)).to(torch.float64)).sum().item())
    return (1j ** (bin(x & z).count("1") % 4)) * r


def _exact_model(case, seed):
    p, x, t = (v.astype(np.float64) for v in _model_inputs(case, seed))
    cut = np.cumsum([0, 1024, 64, 4096, 64, 64, 1])
    w1, b1, w2, b2, w3, b3 = (p[cut[i]:cut[i + 1]] for i in range(6))
    w1, w2 = w1.reshape(64, 16), w2.reshape(64, 64)
    h1 = np.maximum(x @ w1.T + b1, 0)
    h2 = np.maximum(h1 @ w2.T + b2, 0)
    y = h2 @ w3 + b3[0]
    dy = 2.0 * (y - t) / len(t)
    d2 = dy[:, None] * w3 * (h2 > 0)
    d1 = (d2 @ w2) * (h1 > 0)
    grad = np.concatenate([(d1.T @ x).ravel(), d1.sum(0), (d2.T @ h1).ravel(), d2.sum(0), h2.T @ dy, [dy.sum()]])
    return {"y": y, "grad": grad, "loss": float(np.mean((y - t) ** 2))}


def exact(case, seed):
    kind = case["kind"]
    if kind == "model":
        return _exact_model(case, seed)
    if kind == "batch":
        ns, desc = _batch_circuits(case, seed)
        if sum(len(d) for d in desc) > 100000:
            return None
        parts = []
        for n, d in zip(ns, desc):
            parts.append(_simulate(_zero(n), n, d))
            if n < 5:
                parts.append(torch.zeros(32 - (1 << n), dtype=torch.complex128, device=DEV))
        return torch.cat(parts)
    n = case["n"]
    if kind == "readout":
        v = _random_state(case, seed).to(torch.complex128)
        p = torch.view_as_real(v).square().sum(-1)
        return {"norm2": float(p.sum()), "words": np.array([_expval(v, n, x, z) for x, z in _words(case, seed, case["words"])]), "shots": None, "probs": p}
    if kind == "ansatz":
        v = _simulate(_zero(n), n, _hea(_rng(case, seed), n, case["depth"]))
        return {"state": v, "words": np.array([_expval(v, n, x, z) for x, z in _words(case, seed, case["terms"])])}
    if case["circuit"] == "qft" and not case.get("resume"):
        y = torch.arange(1 << n, device=DEV, dtype=torch.int64)
        t = ((y * _basis(case, seed)) & ((1 << n) - 1)).to(torch.float64) * (TWO_PI / (1 << n))
        return torch.polar(torch.full_like(t, 2.0 ** (-n / 2)), t)
    v = _random_state(case, seed).to(torch.complex128) if (case.get("resume") or kind == "host") else _zero(n)
    v = _simulate(v, n, _circuit(case, seed))
    return v.cpu() if kind == "host" else v
