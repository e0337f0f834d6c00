"""complex128 gates in block fixed point (csrc/fixed64.cuh): ranges, exact cases and the FP64 paths
beside it, per-gate and blocked, against the oracle."""
import numpy as np
import pytest

import circuitgen as cg
from oracle import sim

pytestmark = pytest.mark.gpu

# (n, plan options); None: the per-gate path
PATHS = [(7, None), (11, None), (6, dict(chunk_bits=4)), (9, dict(chunk_bits=6)), (14, dict(chunk_bits=12)),
         (13, dict(chunk_bits=10, gather_pinned=4)), (13, dict(chunk_bits=8, diag_outside=1))]


@pytest.fixture(scope="module")
def sv():
    import paper_2102_02957_gb300 as m
    return m


def mixed(n, seed):
    return cg.random_layers(n, 2, seed) + cg.quantum_volume(n, 1, seed) + cg.hea(n, 1, seed, 0) + cg.qft(n, with_swaps=False)


def run(sv, n, desc, opts, start):
    gates = sv.make_gates(desc)
    st = sv.StateVector(n, "c128")
    st.set_state(start)
    st.apply(gates, sv.Plan(n, gates, **opts) if opts is not None else None)
    return st.get_state()


def bound(desc, start):
    """A gate's output component is a sum of at most 8 products of factors of modulus <= 1: FP64 is
    off by at most 8 * 2^-53 * 2 max|x| per gate; gates keep 2-norms, so the sum over gates of the
    2-norm bounds every component.  Both sides round: twice that."""
    return 2 * len(desc) * 16 * 2.0 ** -53 * np.linalg.norm(start)


@pytest.mark.parametrize("n,opts", PATHS)
@pytest.mark.parametrize("scale,spread", [(1.0, 0), (1.0, 40), (2.0 ** -900, 0), (2.0 ** -990, 0), (2.0 ** 1010, 0)])
def test_scaled_states(sv, n, opts, scale, spread):
    rng = np.random.default_rng(n)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    start = start / np.linalg.norm(start) * 10.0 ** -rng.uniform(0, spread, 1 << n) if spread else start / np.linalg.norm(start)
    desc = mixed(n, 3)
    want = sim.apply(start.astype(np.complex128).copy(), n, desc)  # scales by powers of two are exact
    got = run(sv, n, desc, opts, start * scale) / scale
    floor = 2.0 ** -1074 / scale * 64 * len(desc) if scale < 2.0 ** -950 else 0.0  # subnormal steps
    assert np.abs(got - want).max() <= bound(desc, start) + floor


@pytest.mark.parametrize("n,opts", PATHS)
def test_exchanges_and_signs_are_exact(sv, n, opts):
    rng = np.random.default_rng(7)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    desc = [("x", (q,), ()) for q in range(0, n, 2)]
    for q in range(n - 1):
        desc += [("cx", (q, q + 1), ()), ("cx", (q + 1, q), ()), ("cz", (q, q + 1), ()), ("z", (q,), ())]
    perm = np.eye(4)[[2, 0, 3, 1]]
    desc.append(("unitary", (0, n - 1), (perm.astype(np.complex128),)))
    want = sim.apply(start.copy(), n, desc)
    assert np.array_equal(run(sv, n, desc, opts, start), want)
    zero = np.zeros(1 << n, dtype=np.complex128)
    assert np.array_equal(run(sv, n, mixed(n, 5), opts, zero), zero)


@pytest.mark.parametrize("n,opts", PATHS[:5])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_amplitudes_stay_in_their_groups(sv, n, opts, bad):
    rng = np.random.default_rng(1)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    desc = [("u3", (1,), (0.7, 1.1, 2.3)), ("unitary", (0, 2), (cg.haar_unitary(rng),))]
    want = sim.apply(start.copy(), n, desc)
    hit = 5
    start[hit] = complex(bad, 0.25)
    got = run(sv, n, desc, opts, start)
    reached = (np.arange(1 << n) | 7) == (hit | 7)
    assert not np.isfinite(got[reached]).any()
    assert np.abs(got[~reached] - want[~reached]).max() <= bound(desc, start[~reached])


@pytest.mark.parametrize("n,opts", PATHS[:6])
def test_non_unitary_gates_stay_fp64(sv, n, opts):
    rng = np.random.default_rng(2)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    big = 40.0 * (rng.standard_normal((4, 4)) + 1j * rng.standard_normal((4, 4)))
    one = 1e-3 * (rng.standard_normal((2, 2)) + 1j * rng.standard_normal((2, 2)))
    desc = [("unitary", (n - 1, 0), (big,)), ("unitary", (1,), (one,)), ("u3", (0,), (0.3, 0.2, 0.1))]
    want = sim.apply(start.copy(), n, desc)
    got = run(sv, n, desc, opts, start)
    # norms grow by at most ||big|| ||one||; 8 products of 2^-53 each per gate, on both sides
    scale = np.linalg.norm(big, 2) * np.linalg.norm(one, 2) * np.linalg.norm(start)
    assert np.abs(got - want).max() <= 2 * 3 * 16 * 2.0 ** -53 * scale


@pytest.mark.parametrize("n,opts", [(13, dict(chunk_bits=6, diag_outside=1)), (15, dict(chunk_bits=10, diag_outside=1)),
                                    (16, dict(chunk_bits=12, diag_outside=1)), (15, dict(chunk_bits=9, gather_pinned=4, diag_outside=1)),
                                    (14, dict(chunk_bits=5, diag_outside=1))])
@pytest.mark.parametrize("kind", ["qft", "between_dense", "signs"])
def test_merged_outside_diagonals(sv, n, opts, kind):
    """Runs of diagonals from outside the chunk become one per chunk; they may pass diagonal gates and
    gates on other bits, not dense gates or exchanges on theirs."""
    rng = np.random.default_rng(n)
    if kind == "qft":
        desc = cg.qft(n)
    elif kind == "signs":
        desc = [("cz", (int(a), int(b)), ()) for a, b in (rng.choice(n, 2, replace=False) for _ in range(60))]
    else:
        desc = []
        for _ in range(40):
            a, b = (int(v) for v in rng.choice(n, 2, replace=False))
            desc += [("cp", (a, b), (float(rng.uniform(0, 6)),)), ("rz", (a,), (float(rng.uniform(0, 6)),)),
                     ("cp", (b, n - 1 - b if n - 1 - b != b else (b + 1) % n), (0.4,))]
            desc.append([("u3", (a,), (0.3, 0.2, 0.1)), ("cx", (b, a), ()), ("x", (b,), ()), ("ry", (b,), (0.7,))][int(rng.integers(4))])
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    want = sim.apply(start.copy(), n, desc)
    got = run(sv, n, desc, opts, start)
    if kind == "signs":
        assert np.array_equal(got, want)
    else:
        assert np.abs(got - want).max() <= bound(desc, start)


@pytest.mark.parametrize("n,opts", [(6, dict(chunk_bits=4)), (9, dict(chunk_bits=5)), (14, dict(chunk_bits=13)), (14, dict(chunk_bits=12, seg_bits=5)),
                                    (13, dict(chunk_bits=9, gather_pinned=4)), (13, dict(chunk_bits=8, diag_outside=1))])
@pytest.mark.parametrize("kind", ["pairs", "everything"])
def test_fused_complex64_gates(sv, n, opts, kind):
    """Fused records of complex64 sections: every kind of gate before and after every other, same and
    different pairs in both orders, non-unitary matrices among them."""
    rng = np.random.default_rng(n + len(kind))
    desc = []
    for _ in range(60):
        a, b = (int(v) for v in rng.choice(n if kind == "everything" else 4, 2, replace=False))
        desc.append([("u3", (a,), (0.3, 0.2, 0.1)), ("x", (a,), ()), ("rz", (a,), (0.4,)), ("cx", (a, b), ()), ("cz", (a, b), ()),
                     ("cp", (a, b), (0.5,)), ("unitary", (a, b), (cg.haar_unitary(rng),)), ("h", (b,), ()),
                     ("unitary", (a, b), (np.eye(4, dtype=np.complex128)[[1, 2, 3, 0]],)),
                     ("unitary", (a,), (np.array([[0.9, 0.1j], [0.2, 1.1]]),))][int(rng.integers(10))])
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    start = (start / np.linalg.norm(start)).astype(np.complex64)
    want = sim.apply(start.astype(np.complex128), n, desc)
    gates = sv.make_gates(desc)
    st = sv.StateVector(n, "c64")
    st.set_state(start)
    st.apply(gates, sv.Plan(n, gates, **opts))
    # per gate 8 products of 2^-24 each, on norms that the non-unitary gates change by at most 1.2
    grown = 1.2 ** sum(1 for k, q, p in desc if k == "unitary" and len(q) == 1)
    assert np.abs(st.get_state() - want).max() <= len(desc) * 16 * 2.0 ** -24 * grown
