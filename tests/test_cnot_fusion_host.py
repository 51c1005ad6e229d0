"""CNOTs fused as H . CZ . H with the Hadamards multiplied into the neighbouring single-qubit
runs of the target: the compiled plan, executed on the host, against the oracle (no GPU), over
the shapes in which a CNOT does and does not have such runs beside it."""
import numpy as np
import pytest
from test_plan_emulator_host import check, emulator  # noqa: F401  (the fixture)

from workloads import circuits as wc

G = wc.Gate


def chain(n, rng, ends):
    """Sequences of CNOTs onto one target (one to four, nothing in between), with Haar gates, an RX, a
    diagonal gate, another multi-qubit gate or nothing on the target before and after."""
    c = []
    for q in range(n):
        c.append(G("U1", (q,), matrix=wc.haar_2x2(rng)))
    for r in range(12):
        t, *ctl = [int(x) for x in rng.permutation(n)[:5]]
        for side in range(2):
            k = ends[int(rng.integers(len(ends)))]
            if k == "haar":
                c.append(G("U1", (t,), matrix=wc.haar_2x2(rng)))
            elif k == "h":
                c.append(G("H", (t,)))
            elif k == "rx":
                c.append(G("RX", (t,), param=0.7 + r))
            elif k == "rz":
                c.append(G("RZ", (t,), param=0.3 + r))
            elif k == "cz":
                c.append(G("CZ", (ctl[0], t)))
            elif k == "ctl":
                c.append(G("CNOT", (t, ctl[1])))
            if side == 0:
                c += [G("CNOT", (q, t)) for q in ctl[: 1 + int(rng.integers(4))]]
    return c


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("ends", [("haar",), ("h",), ("haar", "none", "h"), ("rx", "rz", "haar"),
                                  ("cz", "ctl", "haar", "none")], ids="-".join)
def test_cnot_sequences(emulator, dtype, ends):  # noqa: F811
    n = 9
    circ = chain(n, np.random.default_rng(len(ends)), ends)
    for tile in (6, 9):
        got, _ = emulator(n, circ, mode="tile", dtype=dtype, tile_bits=tile)
        check(got, circ, n)
