"""CNOTs between gates that only move amplitudes and turn their phases (X, Y, Z, S, and matrices of that kind):
every step of the compiled plan is exact, so the state it leaves, executed on the host (no GPU), is the
oracle's to the last bit.  Products of several such gates are split with the square root of their
determinant, which is exact for 1 and -1; S, of determinant i, therefore stands alone in its run."""
import numpy as np
import pytest
from test_plan_emulator_host import MODES, emulator  # noqa: F401  (the fixture)

from oracle import sv
from workloads import circuits as wc

G = wc.Gate
TURNS = [np.array([[0, -1], [1, 0]]), np.array([[0, -1], [-1, 0]]), np.diag([1j, 1j])]   # determinant 1 or -1


def reversible_circuit(n, layers, seed, kinds):
    """One or two gates of the kinds on every qubit (one where S is among them), then CNOTs on a random matching
    (n even: every qubit's run ends with the layer)."""
    rng = np.random.default_rng(seed)
    c = []
    for _ in range(layers):
        for q in range(n):
            for _ in range(1 if "S" in kinds else 1 + int(rng.integers(2))):
                k = kinds[int(rng.integers(len(kinds)))]
                c.append(G("U1", (q,), matrix=TURNS[int(rng.integers(3))]) if k == "U1" else G(k, (q,)))
        s = [int(q) for q in rng.permutation(n)]
        c += [G("CNOT", (s[2 * i], s[2 * i + 1])) for i in range(n // 2)]
    return c


KINDS = [("Y",), ("X", "Y", "Z"), ("X", "Y", "Z", "S"), ("U1", "X")]


@pytest.mark.parametrize("dtype,arith", MODES)
@pytest.mark.parametrize("kinds", KINDS, ids="-".join)
@pytest.mark.parametrize("n,tile", [(8, 8), (10, 6)])
def test_exact_states(emulator, dtype, arith, n, tile, kinds):  # noqa: F811
    circ = reversible_circuit(n, 40, n + len(kinds), kinds)
    got, _ = emulator(n, circ, mode="tile", dtype=dtype, arith=arith, tile_bits=tile)
    assert np.array_equal(got, sv.simulate(n, circ))
