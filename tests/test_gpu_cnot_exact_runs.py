"""GPU: circuits of moves and quarter turns with CNOTs leave the oracle's state to the last bit, single plan
and batch (products with 0, 1 and -1 and sums with 0 are exact in every arithmetic)."""
import numpy as np
import pytest
from test_cnot_exact_runs_host import KINDS, reversible_circuit

from oracle import sv

pytestmark = pytest.mark.gpu

qs = pytest.importorskip("paper_2010_09746_gb300")


@pytest.mark.parametrize("dtype,arith", [("c128", "df"), ("c128", "f64"), ("c64", "auto")])
@pytest.mark.parametrize("n", [8, 14])
def test_exact_states(dtype, arith, n):
    circs = [reversible_circuit(n, 40, n + len(k), k) for k in KINDS]
    refs = [sv.simulate(n, c) for c in circs]
    for c, ref in zip(circs, refs):
        st = qs.State(n, dtype, arith=arith)
        st.execute(qs.compile(n, c, mode="tile", dtype=dtype, arith=arith))
        assert np.array_equal(st.amplitudes(), ref)
    if arith != "f64":
        b = qs.Batch([(n, c) for c in circs], dtype=dtype)
        b.run()
        assert all(np.array_equal(b.amplitudes(i), refs[i]) for i in range(len(circs)))
