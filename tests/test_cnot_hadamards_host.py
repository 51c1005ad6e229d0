"""The Hadamards that CNOTs bring into their neighbouring runs when they fuse as H . CZ . H: next to a
caller's Hadamard they cancel to the last bit, and over many CNOTs they scale the state neither up nor
down.  The compiled plan, executed on the host (no GPU)."""
import numpy as np
import pytest
from test_plan_emulator_host import check, emulator  # noqa: F401  (the fixture)

from workloads import circuits as wc

G = wc.Gate
R = 1 / np.sqrt(2.0)   # the double below 1 / sqrt 2; sqrt(0.5) is the one above


@pytest.mark.parametrize("arith", ["df", "f64"])
@pytest.mark.parametrize("r", [None, R, np.sqrt(0.5)])
def test_hadamards_beside_a_cnot_cancel(emulator, arith, r):  # noqa: F811
    """H CNOT H on a target is a CZ and nothing else: 200 of them leave a basis state exactly."""
    h = G("H", (1,)) if r is None else G("U1", (1,), matrix=r * np.array([[1, 1], [1, -1]]))
    circ = [G("X", (0,))] + 200 * [h, G("CNOT", (0, 1)), h, G("CNOT", (2, 0))]
    got, _ = emulator(3, circ, mode="tile", dtype="c128", arith=arith)
    want = np.zeros(8)
    want[1] = 1
    assert np.array_equal(got, want)


@pytest.mark.parametrize("arith", ["df", "f64"])
@pytest.mark.parametrize("n,layers", [(2, 1200), (6, 400)])
def test_norm_does_not_drift(emulator, arith, n, layers):  # noqa: F811
    """1200 CNOTs between Haar gates.  Rounded factors 1 / sqrt 2 would add 1200 x 4 x 6.8e-17 = 3.3e-13 to the
    squared norm; roundings to either side (2 x 1.1e-16 for each of some 2400 products and the as many
    updates, as a random walk) stay below 2e-14."""
    circ = wc.haar_cnot_circuit(n, layers, seed=n)
    got, _ = emulator(n, circ, mode="tile", dtype="c128", arith=arith)
    check(got, circ, n)
    assert abs(np.vdot(got, got).real - 1) <= 1e-13
