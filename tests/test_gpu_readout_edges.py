"""Readouts at the edges: Pauli words that cancel, zeros, subnormals and infinities among the amplitudes, many
handles, sampling beside long runs of zeros."""
import numpy as np
import pytest

import circuitgen as cg
from oracle import sim

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    import paper_2102_02957_gb300 as m
    return m


def state(sv, v, dtype):
    st = sv.StateVector(int(np.log2(len(v))), dtype)
    st.set_state(v.astype(np.complex64 if dtype == "c64" else np.complex128))
    return st


def words(n, seed):
    rng = np.random.default_rng(seed)
    out = [(0, 0), (0, 1), (1, 0), (1, 1), (0, (1 << n) - 1), ((1 << n) - 1, 0), (1 << (n - 1), 1 << (n - 1))]
    return out + [tuple(int(v) for v in rng.integers(0, 1 << n, 2)) for _ in range(6)]


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 5, 8, 9, 13, 18])
@pytest.mark.parametrize("kind", ["complex", "real", "turned"])
def test_both_entry_points_return_one_value(sv, dtype, n, kind):
    """Real states cancel under words with an odd number of Y's, and so do real states times a phase (kind turned),
    up to rounding: the two entry points agree in every bit all the same."""
    rng = np.random.default_rng(n)
    v = rng.standard_normal(1 << n) + (1j * rng.standard_normal(1 << n) if kind == "complex" else 0)
    v = v / np.linalg.norm(v) * (np.exp(0.7j) if kind == "turned" else 1)
    st = state(sv, v, dtype)
    back = st.get_state().astype(np.complex128)
    for x, z in words(n, n):
        got, also = st.expval_pauli(x, z), st.expval_pauli_noalloc(x, z)
        assert (got.real, got.imag) == (also.real, also.imag), (x, z, got, also)
        # 2^n terms of 4 products: one rounding each and the sum's, at most log2(2^n) deep a block and 2^11 in sequence
        assert abs(got - sim.expval_pauli(back, x, z)) <= (1 << 11) * 4 * 2.0 ** -53


def edges(n, dtype):
    """Zeros of both signs, subnormals, the smallest and largest normal numbers, in every component."""
    rng = np.random.default_rng(n)
    f = np.float32 if dtype == "c64" else np.float64
    tiny, sub = np.finfo(f).tiny, np.finfo(f).smallest_subnormal
    pool = np.array([0.0, -0.0, sub, -3 * sub, tiny, -tiny, tiny * 1.5, 0.7, -1.3, 1e-20, 2.0 ** 30], dtype=f)
    v = np.empty(1 << n, dtype=np.complex64 if dtype == "c64" else np.complex128)
    v.real, v.imag = rng.choice(pool, 1 << n), rng.choice(pool, 1 << n)
    return v


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 4, 11, 15])
def test_zeros_and_subnormals(sv, dtype, n):
    v = edges(n, dtype)
    st = state(sv, v, dtype)
    re, im = v.real.astype(np.float64), v.imag.astype(np.float64)
    p = re * re + im * im
    # two roundings of an exact product's sum; sums of 2^n of them, the largest 2^60
    assert np.all(np.abs(st.probabilities() - p) <= 2 * 2.0 ** -53 * p + 2.0 ** -1074)
    assert abs(st.norm2() - p.sum()) <= (1 << n) * 2.0 ** -53 * p.sum()
    w = v.astype(np.complex128)
    for x, z in words(n, 5):
        x, z = x & ((1 << n) - 1), z & ((1 << n) - 1)
        assert abs(st.expval_pauli(x, z) - sim.expval_pauli(w, x, z)) <= (1 << n) * 4 * 2.0 ** -53 * p.sum()


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_amplitudes_show(sv, dtype, bad):
    n = 12
    v = edges(n, dtype)
    v[77] = complex(0.5, bad)
    st = state(sv, v, dtype)
    assert not np.isfinite(st.norm2())
    p = st.probabilities()
    assert not np.isfinite(p[77]) and np.count_nonzero(~np.isfinite(p)) == 1
    assert not np.isfinite(st.expval_pauli(0, 5).real)


def test_more_handles_than_result_slots(sv):
    """Handles beyond the pool of pinned result words read through device memory, and slots are given back."""
    for _ in range(2):
        hs = [sv.StateVector(3, "c64") for _ in range(520)]
        for k, h in enumerate(hs):
            h.init_basis(k % 8)
        for k, h in enumerate(hs):
            assert h.norm2() == 1.0
            assert h.expval_pauli(0, 1) == (-1.0 if k & 1 else 1.0)
            assert h.sample(3, k).tolist() == [k % 8] * 3
        for h in hs:
            h.close()


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 3, 9, 10, 11, 16, 21])
def test_sampling_among_zeros(sv, dtype, n):
    """Amplitudes in a few places, whole ranges and blocks of ranges empty: every shot is one of them, and the
    one that the oracle's inverse CDF finds unless its target is within rounding of a boundary."""
    rng = np.random.default_rng(n)
    at = np.unique(np.concatenate([[0, (1 << n) - 1], rng.integers(0, 1 << n, 6)]))
    v = np.zeros(1 << n, dtype=np.complex128)
    v[at] = rng.uniform(0.2, 1.0, len(at)).astype(np.float32)
    st = state(sv, v, dtype)
    shots, seed = 4000, 9
    got = st.sample(shots, seed).astype(np.int64)
    cum = np.cumsum(np.abs(v[at]) ** 2)
    t = np.array([sim.uniform(seed, s) for s in range(shots)]) * cum[-1]
    want = at[np.searchsorted(cum, t, side="right")]
    near = np.min(np.abs(cum[None, :] - t[:, None]), axis=1) <= 64 * 2.0 ** -53 * cum[-1]
    assert np.isin(got, at).all()
    assert np.array_equal(got[~near], want[~near])
