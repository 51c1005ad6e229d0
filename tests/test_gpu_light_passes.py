"""GPU: complex64 passes without moves give the same bits from either side of the 2^14 tiles where they change
kernels (the batched kernel as the common reference), and the oracle's amplitudes."""
import numpy as np
import pytest

from oracle import sv
from workloads import circuits as wc

pytestmark = pytest.mark.gpu

qs = pytest.importorskip("paper_2010_09746_gb300")


@pytest.mark.parametrize("n", [18, 19])
def test_same_bits_as_the_batched_kernel(n):
    circs = [wc.rzrx_cz_circuit(n, 4, n), wc.rzrx_cz_circuit(n, 3, n) + [wc.Gate("CNOT", (0, 1)), wc.Gate("RX", (1,), param=0.5)]]
    b = qs.Batch([(n, c) for c in circs], dtype="c64", tile_bits=5, low_bits=2)
    b.run()
    for i, c in enumerate(circs):
        st = qs.State(n, "c64")
        st.execute(qs.compile(n, c, mode="tile", dtype="c64", tile_bits=5, low_bits=2, dense=False))
        got = st.amplitudes()
        assert got.tobytes() == b.amplitudes(i).tobytes()
        assert np.abs(got - sv.simulate(n, c)).max() <= 1e-5
