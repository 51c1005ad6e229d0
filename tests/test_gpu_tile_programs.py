"""GPU: tile passes whose program travels in the kernel parameters give the bits of those that read it
from device arrays (the batched kernel does), and the oracle's amplitudes: circuits whose passes all
fit, passes with ops that have no such form (a dense block, a SWAP), a program larger than the
parameter space, and states on either side of one tile per SM."""
import numpy as np
import pytest

from oracle import sv
from workloads import circuits as wc

pytestmark = pytest.mark.gpu

qs = pytest.importorskip("paper_2010_09746_gb300")

G = wc.Gate


def circuits(n, seed):
    rng = np.random.default_rng(seed)
    c = []   # X, controlled phases and RX in runs that stay apart (CNOT on either side of an RX)
    for _ in range(40):
        a, b = [int(x) for x in rng.choice(n, 2, replace=False)]
        c += [G("RX", (a,), param=float(rng.uniform(0, 6))), G("CNOT", (a, b)),
              G("CP", (b, a), param=float(rng.uniform(0, 6))), G("X", (b,)), G("CZ", (a, b))]
    return [wc.mixed_batch_circuit(n, 6, rng), wc.rzrx_cz_circuit(n, 8, seed), wc.qft_circuit(n), wc.qft_like_circuit(n),
            wc.paper_random_circuit(n, 0.4, seed), wc.single_qubit_run_circuit(n, 6, seed), c,
            wc.random_mixed_circuit(n, 60, seed), wc.haar_cnot_circuit(n, 160 if n <= 9 else 4, seed)]


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,tile", [(6, 0), (9, 0), (12, 0), (13, 8), (15, 9), (19, 0), (20, 0)])
def test_same_bits_as_the_batched_kernel(dtype, n, tile):
    circs = circuits(n, n)
    b = qs.Batch([(n, c) for c in circs], dtype=dtype, tile_bits=tile)
    b.run()
    for i, c in enumerate(circs):
        st = qs.State(n, dtype)
        st.execute(qs.compile(n, c, mode="tile", dtype=dtype, tile_bits=tile, dense=False))
        got = st.amplitudes()
        assert got.tobytes() == b.amplitudes(i).tobytes(), i
        if n <= 15:
            assert np.abs(got - sv.simulate(n, c)).max() <= (1e-12 if dtype == "c128" else 1e-5), i
