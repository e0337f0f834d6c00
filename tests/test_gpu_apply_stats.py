"""Statistics of per-gate circuits count what their sweeps move and launch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    import paper_2102_02957_gb300 as m
    return m


@pytest.mark.parametrize("dtype,amp", [("c64", 8), ("c128", 16)])
def test_bytes_and_launches(sv, dtype, amp):
    n = 10
    full = 2 * (1 << n) * amp
    one = np.eye(2, dtype=np.complex128)
    # on qubit 0 complex64 sweeps everything; shares of the state elsewhere
    for desc, share, launches in [([("h", (3,), ())], 1, 1), ([("cx", (4, 2), ())], 0.5, 1), ([("cz", (4, 2), ())], 0.25, 1),
                                  ([("cp", (4, 2), (0.3,))], 0.25, 1), ([("rz", (5,), (0.3,))], 1, 1), ([("swap", (4, 2), ())], 0.5, 1),
                                  ([("unitary", (3,), (one,))], 0, 0), ([("cx", (4, 0), ())], 1 if dtype == "c64" else 0.5, 1),
                                  ([("h", (3,), ()), ("cz", (4, 2), ()), ("unitary", (3,), (one,))], 1.25, 2)]:
        st = sv.StateVector(n, dtype)
        st.init_basis(0)
        st.apply(sv.make_gates(desc))
        s = st.stats()
        assert (s.algorithmic_bytes, s.kernel_launches, s.sweeps_gate) == (share * full, launches, len(desc)), desc
        st.close()
