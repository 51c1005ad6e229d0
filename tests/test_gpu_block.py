"""GPU: general blocks held in registers (one to five qubits) against the FP64 oracle, where the
kernel changes its way of loading: states too small for a warp's 32 groups, target bits on
either side of the line between the two ways, low and scattered targets, and a control."""
import numpy as np
import pytest

from oracle import sv
from workloads import circuits as wc

pytestmark = pytest.mark.gpu

qs = pytest.importorskip("paper_2010_09746_gb300")

MODES = [("c64", "auto"), ("c128", "df"), ("c128", "f64")]
TOL = {"c64": 2e-6, "c128": 1e-13}   # a few roundings of 2^k terms of a unit vector


def random_state(n, rng):
    v = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    return v / np.linalg.norm(v)


@pytest.mark.parametrize("dtype,arith", MODES)
@pytest.mark.parametrize("n,qubits", [
    (1, [0]), (2, [1, 0]), (5, [2, 0, 4, 1, 3]), (6, [5]), (7, [0, 1]), (9, [3, 0, 1, 2]), (10, [4, 3, 2, 1, 0]),
    (11, [9, 2, 5]), (12, [1, 11]), (13, [3, 12, 7, 5]), (14, [13, 0, 6, 2, 9]), (14, [2, 3]), (15, [3, 4, 5, 6, 7]),
    (13, [12, 11, 10, 9, 8, 7])])
def test_blocks(dtype, arith, n, qubits):
    rng = np.random.default_rng(n + len(qubits))
    st = qs.State(n, dtype, arith=arith)
    st.set_dense_path("cuda_cores")
    psi = random_state(n, rng).astype(st.np_dtype)
    o = sv.OracleState(n, psi.astype(np.complex128))
    st.set_amplitudes(psi)
    for k in range(2):   # the same qubits in both orders
        U = wc.haar_unitary(1 << len(qubits), rng)
        q = qubits[:: 1 - 2 * k]
        st.apply_dense(U, q)
        o.apply_dense(U, q)
    assert np.abs(st.amplitudes() - o.psi).max() <= TOL[dtype]


@pytest.mark.parametrize("dtype,arith", MODES)
@pytest.mark.parametrize("n,c,t", [(2, 0, 1), (6, 0, 5), (7, 6, 0), (8, 2, 1), (9, 0, 3), (12, 5, 11), (12, 11, 2)])
def test_controlled(dtype, arith, n, c, t):
    rng = np.random.default_rng(7 * n + c)
    st = qs.State(n, dtype, arith=arith)
    psi = random_state(n, rng).astype(st.np_dtype)
    st.set_amplitudes(psi)
    U = wc.haar_unitary(2, rng)
    st.apply_controlled(U, c, t)
    i = np.arange(1 << n)
    a, b = psi[i & ~(1 << t)].astype(np.complex128), psi[i | (1 << t)].astype(np.complex128)
    want = np.where((i >> t) & 1, U[1, 0] * a + U[1, 1] * b, U[0, 0] * a + U[0, 1] * b)
    want = np.where((i >> c) & 1, want, psi)
    assert np.abs(st.amplitudes() - want).max() <= TOL[dtype]
