"""A plan keeps the register groups of its sections: used again with other angles, by several threads at a
time, for both types and engines, against the oracle."""
import threading

import numpy as np
import pytest

import circuitgen as cg
from oracle import sim

pytestmark = pytest.mark.gpu

PLANS = [dict(chunk_bits=11), dict(chunk_bits=8), dict(chunk_bits=11, diag_outside=1), dict(chunk_bits=11, gather_pinned=4),
         dict(chunk_bits=12, gather_pinned=4, use_tc=1)]


@pytest.fixture(scope="module")
def sv():
    import paper_2102_02957_gb300 as m
    return m


def circuit(n, seed):
    """The same structure for every seed."""
    r = np.random.default_rng(seed)
    out = []
    for layer in range(3):
        out += [("u3", (q,), tuple(r.uniform(0, 6, 3))) for q in range(n)]
        out += [("cp", (q, (q + 5) % n), (float(r.uniform(0, 6)),)) for q in range(n)]
        out += [("cx", (q, q + 1), ()) for q in range(layer, n - 1, 2)]
    return out + [("cp", (q, n - 1), (float(r.uniform(0, 6)),)) for q in range(n - 1)]


@pytest.mark.parametrize("opts", PLANS)
def test_one_plan_for_all(sv, opts):
    n = 14
    plan = sv.Plan(n, sv.make_gates(circuit(n, 0)), **opts)
    errors = []

    def work(k):
        try:
            import torch
            dtype = "c64" if k % 2 else "c128"
            with torch.cuda.stream(torch.cuda.Stream()):
                st = sv.StateVector(n, dtype, stream=torch.cuda.current_stream())
                for seed in range(3):
                    desc = circuit(n, 10 * k + seed)
                    st.init_basis(k)
                    st.apply(sv.make_gates(desc), plan)
                    want = sim.apply(sim.basis_state(n, k), n, desc)
                    err = np.abs(st.get_state() - want).max()
                    # 16 products of a unit per gate, on a state of norm 1
                    assert err <= len(desc) * 16 * (2.0 ** -24 if dtype == "c64" else 2.0 ** -53), (k, seed, err)
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_per_gate_sweeps_between_other_work(sv):
    """Per-gate launches overlap their predecessors' ends: copies and another stream's kernels before and after them."""
    import torch
    n, desc = 18, cg.random_layers(18, 2, 3)
    gates = sv.make_gates(desc)
    rng = np.random.default_rng(0)
    start = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    want = sim.apply(start.copy(), n, desc)
    src = torch.from_numpy(start).cuda()
    buf, out = torch.empty_like(src), []
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        st = sv.StateVector(n, "c128", buffer=buf, stream=s)
        for k in range(8):
            with torch.cuda.stream(other):
                noise = torch.randn(1 << 20, device="cuda").sin_()  # noqa: F841
            buf.copy_(src)
            if k % 2:
                buf.mul_(2.0)
            st.apply(gates)
            out.append(buf.clone())
            buf.zero_()
    torch.cuda.synchronize()
    bound = 2 * len(desc) * 18 * 2.0 ** -53 * np.linalg.norm(start)
    for k, o in enumerate(out):
        assert np.abs(o.cpu().numpy() / (2.0 if k % 2 else 1.0) - want).max() <= bound
