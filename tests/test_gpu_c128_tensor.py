"""complex128 sections on the tensor cores (csrc/block_oz.cuh): chunk widths, group counts, several
sweeps per section, amplitude ranges and the FP64 fallback of single chunks, against the oracle."""
import numpy as np
import pytest

import circuitgen as cg
from oracle import sim

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    import paper_2102_02957_gb300 as m
    return m


def run(sv, n, desc, opts, start):
    gates = sv.make_gates(desc)
    st = sv.StateVector(n, "c128")
    st.set_state(start)
    plan = sv.Plan(n, gates, **opts)
    st.apply(gates, plan)
    return st.get_state(), st.stats(), plan.info()


def bound(desc, start):
    """Per gate FP64 is off by at most 8 products of 2^-53 * 2 max|x|, and gates keep 2-norms; per group
    (at most one per gate here) the integer form rounds to 2^-54 of the chunk's largest component and
    U to 2^-55 per entry, 32 of them: less than the same again."""
    return 3 * len(desc) * 16 * 2.0 ** -53 * np.linalg.norm(start)


@pytest.mark.parametrize("n,opts", [(11, dict(chunk_bits=11)), (12, dict(chunk_bits=12)), (13, dict(chunk_bits=13)),
                                    (14, dict(chunk_bits=11)), (15, dict(chunk_bits=12)), (16, dict(chunk_bits=13)),
                                    (15, dict(chunk_bits=12, reserve=1)), (16, dict(chunk_bits=11, gather_pinned=4)),
                                    (17, dict(chunk_bits=12, gather_pinned=5, lookahead=1))])
@pytest.mark.parametrize("kind", ["one", "layers", "volume", "mixed"])
def test_against_oracle(sv, n, opts, kind):
    rng = np.random.default_rng(n)
    desc = {"one": [("h", (n - 1,), ())], "layers": cg.random_layers(n, 2, 4), "volume": cg.quantum_volume(n, 2, 5),
            "mixed": cg.hea(n, 1, 6, 0) + cg.qft(n) + cg.random_layers(n, 1, 7)}[kind]
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    want = sim.apply(start.copy(), n, desc)
    got, _, _ = run(sv, n, desc, opts, start)
    assert np.abs(got - want).max() <= bound(desc, start)


def test_many_groups_take_several_sweeps(sv):
    n = 12
    desc = cg.quantum_volume(n, 8, 1)
    rng = np.random.default_rng(0)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    got, stats, info = run(sv, n, desc, dict(chunk_bits=12), start)
    assert info.n_blocks == 1 and stats.sweeps_block > 1
    assert np.abs(got - sim.apply(start.copy(), n, desc)).max() <= bound(desc, start)


@pytest.mark.parametrize("scale", [2.0 ** -900, 2.0 ** -1000, 2.0 ** 1005])
def test_scaled_states(sv, scale):
    n = 13
    rng = np.random.default_rng(3)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    start /= np.linalg.norm(start)
    desc = cg.random_layers(n, 2, 9)
    want = sim.apply(start.copy(), n, desc)
    got = run(sv, n, desc, dict(chunk_bits=11), start * scale)[0] / scale
    floor = 2.0 ** -1074 / scale * 64 * len(desc) if scale < 2.0 ** -950 else 0.0  # subnormal steps
    assert np.abs(got - want).max() <= bound(desc, start) + floor


def test_chunks_of_zeros_and_of_one_huge_amplitude(sv):
    n = 14
    desc = [("u3", (q,), (0.3 + q, 0.2, 0.1)) for q in range(11)]  # no gate leaves its 11-bit chunk
    start = np.zeros(1 << n, dtype=np.complex128)
    start[5] = 1e200
    start[(1 << 11) + 3] = 1e-200
    start[(3 << 11):(4 << 11)] = 1.0
    want = sim.apply(start.copy(), n, desc)
    got, _, _ = run(sv, n, desc, dict(chunk_bits=11), start)
    for c in range(8):  # each chunk is accurate to its own norm
        part = slice(c << 11, (c + 1) << 11)
        top = max(np.abs(start[part]).max(), 1e-300)  # squares of 1e-200 and 1e200 leave the range
        norm = np.linalg.norm(start[part] / top) * top
        assert np.abs(got[part] - want[part]).max() <= 3 * len(desc) * 16 * 2.0 ** -53 * norm


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_chunk_runs_in_fp64(sv, bad):
    n = 13
    rng = np.random.default_rng(1)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    desc = [("u3", (1,), (0.7, 1.1, 2.3)), ("unitary", (0, 2), (cg.haar_unitary(rng),)), ("cx", (4, 5), ())]
    want = sim.apply(start.copy(), n, desc)
    start[5] = complex(bad, 0.25)
    got, _, _ = run(sv, n, desc, dict(chunk_bits=11), start)
    reached = (np.arange(1 << n) | 7) == 7  # the three dense qubits' coset (bit 4 of index 5 is 0)
    assert not np.isfinite(got[reached]).any()
    assert np.abs(got[~reached] - want[~reached]).max() <= bound(desc, start[~reached])


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,c,share,pinned_host", [(18, 9, 4, True), (20, 10, 8, True), (21, 12, 4, False), (19, 6, 8, True), (20, 11, 16, True)])
def test_host_resident_gathered_passes(sv, dtype, n, c, share, pinned_host):
    """The gathered passes of host-resident states: both types, mapped and pageable host memory, chunk
    widths on either side of the gathered inner plan's."""
    import torch
    desc = cg.random_layers(n, 3, 2) + cg.quantum_volume(n, 1, 3)
    rng = np.random.default_rng(n)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    start /= np.linalg.norm(start)
    want = sim.apply(start.copy(), n, desc)
    gates = sv.make_gates(desc)
    plan = sv.Plan(n, gates, chunk_bits=c)
    ct = np.complex64 if dtype == "c64" else np.complex128
    host = torch.from_numpy(start.astype(ct))
    host = host.pin_memory() if pinned_host else host
    passes = sv.apply_host(n, host, gates, plan, (1 << n) // share * host.element_size(), dtype=dtype)
    info = plan.info()
    assert 1 <= passes < info.n_blocks + info.n_swap_rounds + info.n_unpermute_rounds
    tol = 1e-5 if dtype == "c64" else 1e-12
    assert np.abs(host.numpy() - want).max() <= tol
