"""GPU: register-stage factors that depend on one or two register slots (narrowed phase tables, sign
flips and phases with one control outside the registers, groups of them on one slot), at every
register width and with tiles smaller than the state, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import sv
from workloads import circuits as wc

pytestmark = pytest.mark.gpu

qs = pytest.importorskip("paper_2010_09746_gb300")

G = wc.Gate


def circuit(n, seed, phases):
    """Layers of RX on a few qubits, then controlled phases onto each of them from several others (a
    group on one slot), CZ pairs (sign flips) and lone phases (tables of one and two slots)."""
    rng = np.random.default_rng(seed)
    c = [G("H", (q,)) for q in range(n)]
    for _ in range(4):
        qs_ = [int(q) for q in rng.permutation(n)]
        for q in qs_[:4]:
            c.append(G("RX", (q,), param=float(rng.uniform(0, 6.2))))
        for q in qs_[:2]:
            c += [G("CP", (r, q), param=float(rng.uniform(0, 6.2))) for r in qs_[2: 2 + phases]]
            c.append(G("P", (q,), param=float(rng.uniform(0, 6.2))))
        c += [G("CZ", (qs_[i], qs_[-1 - i])) for i in range(2)]
    return c


@pytest.mark.parametrize("dtype,arith,K", [("c64", "auto", k) for k in (1, 2, 3, 4, 5)] +
                         [("c128", a, k) for a in ("df", "f64") for k in (1, 2, 3, 4)])
@pytest.mark.parametrize("n,tile,phases", [(5, 5, 1), (10, 6, 2), (11, 8, 8), (13, 12, 5)])
def test_factors_on_few_slots(dtype, arith, K, n, tile, phases):
    circ = circuit(n, 100 * n + K, min(phases, n - 2))
    st = qs.State(n, dtype, arith=arith)
    st.execute(qs.compile(n, circ, mode="tile", dtype=dtype, arith=arith, tile_bits=tile, reg_bits=K))
    err = np.abs(st.amplitudes() - sv.simulate(n, circ)).max()
    assert err <= (1e-12 if dtype == "c128" else 1e-5)
