"""complex128 results amplitude by amplitude: states whose amplitudes spread over many orders of magnitude
keep each of them to the accuracy that FP64 gives it, against the oracle."""
import numpy as np
import pytest

import circuitgen as cg
from oracle import sim

pytestmark = pytest.mark.gpu

# (n, plan options); None: the per-gate path.  Sections on the integer pipe (chunks below 11 bits, diagonals from
# outside the chunk), on the tensor cores (11 to 13 bits, contiguous and gathered), in FP64.
PATHS = [(7, None), (12, None), (6, dict(chunk_bits=4)), (9, dict(chunk_bits=6)), (12, dict(chunk_bits=9, gather_pinned=4)),
         (12, dict(chunk_bits=8, diag_outside=1)), (13, dict(chunk_bits=11, diag_outside=1)), (11, dict(chunk_bits=11)),
         (14, dict(chunk_bits=12)), (14, dict(chunk_bits=13)), (14, dict(chunk_bits=11, gather_pinned=4, lookahead=1)),
         (13, dict(chunk_bits=11, fp64_sections=1))]


@pytest.fixture(scope="module")
def sv():
    import paper_2102_02957_gb300 as m
    return m


def run(sv, n, desc, opts, start):
    gates = sv.make_gates(desc)
    st = sv.StateVector(n, "c128")
    st.set_state(start)
    st.apply(gates, sv.Plan(n, gates, **opts) if opts is not None else None)
    return st.get_state()


def magnitudes(n, desc, start):
    """Per amplitude the sum of |products| that make it: the state of |start| under the gates' moduli."""
    w = [(k, qs, p) for k, qs, p in desc]
    return sim.apply(np.abs(start).astype(np.complex128), n, [("unitary", qs, (np.abs(cg_matrix(k, qs, p)).astype(np.complex128),)) for k, qs, p in w]).real


def cg_matrix(kind, qs, params):
    """The gate's matrix in its qubits' own basis, column by column from the oracle."""
    if kind == "unitary":
        return params[0]
    m = len(qs)
    cols = []
    for b in range(1 << m):
        e = np.zeros(1 << m, dtype=np.complex128)
        e[b] = 1
        cols.append(sim.apply(e, m, [(kind, tuple(range(m)), params)]))
    return np.array(cols).T


def spread_states(n):
    rng = np.random.default_rng(n)
    dense = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    one = np.zeros(1 << n, dtype=np.complex128)
    one[0] = 1
    tiny = dense.copy()
    tiny[3::5] *= 1e-10
    tiny[4::7] *= 1e-18
    tiny[1] = 1e-300
    pair = one.copy()
    pair[1:] = 1e-20
    wide = dense * 10.0 ** -rng.uniform(0, 60, 1 << n)
    speck = dense.copy()
    speck[3] *= 1e-18
    speck[5] = 0
    return {"basis": one, "pair": pair, "planted": tiny, "wide": wide, "speck": speck}


def circuits(n):
    return {"phases": [("rz", (q,), (0.3 + q,)) for q in range(n)] + [("cp", (q, q + 1), (0.7,)) for q in range(n - 1)],
            "angles": [("ry", (q,), (1e-6,)) for q in range(n)],
            "steep": [("u3", (q,), (10.0 ** -(q % 4) * 0.9, 0.4, 0.2)) for q in range(n)] + [("cx", (q, q + 1), ()) for q in range(n - 1)],
            "layers": cg.random_layers(n, 2, 5), "volume": cg.quantum_volume(n, 2, 6), "qft": cg.qft(n),
            "cat": [("h", (0,), ())] + [("cx", (q, q + 1), ()) for q in range(n - 1)] + [("u3", (q,), (0.0, 0.3 + q, 0.1)) for q in range(n)] * 3}


@pytest.mark.parametrize("n,opts", PATHS)
@pytest.mark.parametrize("state", ["basis", "pair", "planted", "wide", "speck"])
@pytest.mark.parametrize("circuit", ["phases", "angles", "steep", "layers", "volume", "qft", "cat"])
def test_every_amplitude_is_as_exact_as_in_fp64(sv, n, opts, state, circuit):
    """A gate's output is a sum of at most 8 real products per component: FP64 is off by at most 9 units of 2^-53
    of the sum of their moduli, 18 for both components and their cross terms; both sides round, gate after gate."""
    start, desc = spread_states(n)[state], circuits(n)[circuit]
    want = sim.apply(start.copy(), n, desc)
    got = run(sv, n, desc, opts, start)
    bound = 2 * len(desc) * 18 * 2.0 ** -53 * magnitudes(n, desc, start) + 2.0 ** -1074 * 64 * len(desc)
    worst = np.argmax(np.abs(got - want) - bound)
    assert np.all(np.abs(got - want) <= bound), (worst, got[worst], want[worst], bound[worst])


def test_phases_keep_a_small_amplitude(sv):
    start = np.array([1.0, 1e-20], dtype=np.complex128)
    got = run(sv, 1, [("rz", (0,), (0.8,))], None, start)
    assert abs(got[1] / (1e-20 * np.exp(0.4j)) - 1) <= 8 * 2.0 ** -53


@pytest.mark.parametrize("state", ["planted", "wide"])
@pytest.mark.parametrize("share", [4, 8])
def test_host_resident_states_keep_every_amplitude(sv, state, share):
    import torch
    n = 17
    start, desc = spread_states(n)[state], circuits(n)["steep"]
    gates = sv.make_gates(desc)
    host = torch.from_numpy(start.copy()).pin_memory()
    sv.apply_host(n, host, gates, sv.Plan(n, gates, chunk_bits=11), (1 << n) // share * 16, dtype="c128")
    want = sim.apply(start.copy(), n, desc)
    bound = 2 * len(desc) * 18 * 2.0 ** -53 * magnitudes(n, desc, start) + 2.0 ** -1074 * 64 * len(desc)
    assert np.all(np.abs(host.numpy() - want) <= bound)


@pytest.mark.parametrize("opts", [dict(chunk_bits=8), dict(chunk_bits=11), dict(chunk_bits=12)])
def test_chunks_run_apart(sv, opts):
    """Dense, sparse, empty, non-finite and peaked chunks side by side: each is accurate to itself."""
    n, c = 15, opts["chunk_bits"]
    rng = np.random.default_rng(4)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    parts = start.reshape(-1, 1 << c)
    parts[1] = 0
    parts[2, 1:] = 0
    parts[3, ::3] *= 1e-12
    parts[4] *= 1e-290
    parts[5, 7] = complex(np.inf, 0.5)
    desc = cg.random_layers(c, 3, 2) + cg.quantum_volume(c, 2, 3)  # on the chunk's own qubits
    got = run(sv, n, desc, opts, start).reshape(-1, 1 << c)
    for k in range(len(parts)):
        if k == 5:
            assert not np.isfinite(got[k]).all()
            continue
        want = sim.apply(parts[k].copy(), c, desc)
        bound = 2 * len(desc) * 18 * 2.0 ** -53 * magnitudes(c, desc, parts[k]) + 2.0 ** -1074 * 64 * len(desc)
        assert np.all(np.abs(got[k] - want) <= bound), k


def extended(n, desc, start):
    """The circuit in extended precision (64 or 113 mantissa bits), gate by gate."""
    v = start.astype(np.clongdouble)
    for kind, qs, ps in desc:
        m, d = cg_matrix(kind, qs, ps).astype(np.clongdouble), 1 << len(qs)
        idx = np.arange(1 << n)
        mask = sum(1 << q for q in qs)
        base = idx[(idx & mask) == 0]
        at = [base | sum(((b >> j) & 1) << q for j, q in enumerate(qs)) for b in range(d)]
        old = [v[a] for a in at]
        for r in range(d):
            v[at[r]] = sum(m[r, k] * old[k] for k in range(d))
    return v


@pytest.mark.parametrize("n,opts", [(11, dict(chunk_bits=11)), (12, dict(chunk_bits=12)), (13, dict(chunk_bits=13)), (12, dict(chunk_bits=9))])
@pytest.mark.parametrize("kind", ["layers", "volume", "mixed"])
def test_dense_states_are_no_less_exact_than_in_fp64(sv, n, opts, kind):
    """The root mean square error of a dense state against extended precision: fixed point and digit products
    have finer units than FP64's roundings, so that theirs is the smaller one; one lost digit, product
    or rounding would make it many times larger."""
    rng = np.random.default_rng(n)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    desc = {"layers": cg.random_layers(n, 6, 4), "volume": cg.quantum_volume(n, 5, 5), "mixed": cg.random_layers(n, 3, 7) + cg.qft(n, with_swaps=False)}[kind]
    want = extended(n, desc, start)

    def error(**more):
        d = run(sv, n, desc, dict(opts, **more), start).astype(np.clongdouble) - want
        return float(np.sqrt(np.mean(d.real ** 2 + d.imag ** 2)))

    assert error() <= error(fp64_sections=1)
