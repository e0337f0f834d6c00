"""complex64 register groups on the SIMT path give the bits of their gates applied one after another."""
import numpy as np
import pytest

import circuitgen as cg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    import paper_2102_02957_gb300 as m
    return m


def run(sv, n, descs, start, **opts):
    """The state after each circuit of `descs` in turn, each as sections of a plan of its own."""
    st = sv.StateVector(n, "c64")
    st.set_state(start)
    for d in descs:
        gates = sv.make_gates(d)
        st.apply(gates, sv.Plan(n, gates, **opts))
    return st.get_state()


def circuit(kind, n):
    """On n qubits, few enough for one register group: groups may be cut in another order than the list's."""
    if kind == "layers":
        return cg.random_layers(n, 3, 1)
    if kind == "ansatz":  # real states, whose words with an odd number of Y's vanish
        return cg.hea(n, 3, 2, 0)
    return cg.qft(n, with_swaps=False) + cg.quantum_volume(n, 2, 3) + [("x", (q,), ()) for q in range(n)] + cg.random_layers(n, 1, 4)


@pytest.mark.parametrize("n,opts,on", [(6, dict(chunk_bits=6), (0, 1, 2, 3)), (9, dict(chunk_bits=9), (8, 0, 5, 2)), (13, dict(chunk_bits=13), (11, 12, 3, 7)),
                                       (11, dict(chunk_bits=11, seg_bits=5), (4, 10, 0, 6, 1))])
@pytest.mark.parametrize("kind", ["layers", "ansatz", "mixed"])
def test_a_register_group_has_the_bits_of_its_gates(sv, n, opts, on, kind):
    rng = np.random.default_rng(n)
    start = (rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)).astype(np.complex64)
    desc = [(k, tuple(on[q] for q in qs), p) for k, qs, p in circuit(kind, len(on))]
    assert np.array_equal(run(sv, n, [desc], start, **opts), run(sv, n, [[g] for g in desc], start, **opts))


@pytest.mark.parametrize("desc", [[("x", (1,), ()), ("z", (1,), ())], [("z", (1,), ()), ("x", (1,), ())], [("x", (1,), ()), ("x", (1,), ())],
                                  [("x", (0,), ()), ("z", (0,), ()), ("x", (1,), ()), ("z", (1,), ()), ("cx", (0, 1), ())]])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_exchanges_and_signs_keep_a_non_finite_amplitude_single(sv, desc, bad):
    n = 8
    start = np.ones(1 << n, dtype=np.complex64)
    start[5] = complex(bad, 0.25)
    got = run(sv, n, [desc], start, chunk_bits=n)
    assert np.count_nonzero(~np.isfinite(got)) == 1
