"""complex128 results amplitude by amplitude: states whose amplitudes spread over many orders of magnitude
keep each of them to the accuracy that FP64 gives it, against the oracle."""
import numpy as np
import pytest

import circuitgen as cg
from oracle import sim

pytestmark = pytest.mark.gpu

# (n, plan options); None: the per-gate path
PATHS = [(7, None), (12, None)]


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
    return {"basis": one, "pair": pair, "planted": tiny, "wide": wide}


def circuits(n):
    return {"phases": [("rz", (q,), (0.3 + q,)) for q in range(n)] + [("cp", (q, q + 1), (0.7,)) for q in range(n - 1)],
            "angles": [("ry", (q,), (1e-6,)) for q in range(n)],
            "steep": [("u3", (q,), (10.0 ** -(q % 4) * 0.9, 0.4, 0.2)) for q in range(n)] + [("cx", (q, q + 1), ()) for q in range(n - 1)],
            "layers": cg.random_layers(n, 2, 5), "volume": cg.quantum_volume(n, 2, 6)}


@pytest.mark.parametrize("n,opts", PATHS)
@pytest.mark.parametrize("state", ["basis", "pair", "planted", "wide"])
@pytest.mark.parametrize("circuit", ["phases", "angles", "steep", "layers", "volume"])
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
