"""Long passes whose RX angles all lie near pi (a kicked chain with imperfect pi pulses): the sines that
tangent-form RX drop are just below 1, no cosine among them is large, and the dropped factors are
still absorbed before they leave the range of a float.  The compiled plan, executed on the host (no GPU).

A segment closes by 2^24 of growth, so registers stay below 2^25, and its closing RX keeps entries
(c, s) times at least 2^-24.  The emulator reports the smallest such entry; for double-float plans,
whose c and s are separate entries, that is the one of c, so the bound there carries the circuit's smallest
|cos|."""
import numpy as np
import pytest
from test_plan_emulator_host import MODES, check, emulator  # noqa: F401  (the fixture)

from workloads import circuits as wc

G = wc.Gate


def kicked_chain(n, layers, angle, pair="CZ", seed=0, general=False):
    """RX(angle) on every qubit (general: as a 2x2 matrix between diagonal factors), then the pair gate on
    alternating neighbours of the ring; a tuple of angles is a range to draw from."""
    rng = np.random.default_rng(seed)
    c = []
    for k in range(layers):
        for q in range(n):
            t = float(rng.uniform(*angle)) if isinstance(angle, tuple) else angle
            if general:
                a, b = np.exp(1j * rng.uniform(0, 2 * np.pi, 2))
                r = np.array([[np.cos(t / 2), -1j * np.sin(t / 2)], [-1j * np.sin(t / 2), np.cos(t / 2)]])
                c.append(G("U1", (q,), matrix=np.diag([1, a]) @ r @ np.diag([1, b])))
            else:
                c.append(G("RX", (q,), param=t))
        c += [G(pair, (q, (q + 1) % n)) for q in range(k % 2, n, 2)]
    return c


def min_cos(circ):
    return min(abs(np.cos(g.param / 2)) if g.kind == "RX" else abs(g.matrix[0, 0])
               for g in circ if g.kind in ("RX", "U1"))


@pytest.mark.parametrize("dtype,arith", MODES)
@pytest.mark.parametrize("n,layers,angle,pair,general", [
    (12, 400, 0.85 * np.pi, "CZ", False), (12, 400, (0.85 * np.pi, 1.15 * np.pi), "CZ", False),
    (12, 400, 2.7, "CNOT", False), (10, 400, 3.1, "CZ", False), (10, 400, 2 * np.arccos(0.249), "CZ", False),
    (10, 400, 2.7, "CZ", True), (6, 800, 0.9 * np.pi, "CZ", False), (3, 1600, 0.9 * np.pi, "CZ", False)])
def test_angles_near_pi(emulator, dtype, arith, n, layers, angle, pair, general):  # noqa: F811
    circ = kicked_chain(n, layers, angle, pair, general=general)
    got, _ = emulator(n, circ, mode="tile", dtype=dtype, arith=arith, tile_bits=n)
    check(got, circ, n)
    assert emulator.max_register_abs < 2.0 ** 25, emulator.max_register_abs
    least = 2.0 ** -25 * (min_cos(circ) if arith == "df" else 1.0)
    assert emulator.min_register_scale > least, (emulator.min_register_scale, least)


@pytest.mark.parametrize("dtype,arith", MODES)
def test_rx_alone(emulator, dtype, arith):  # noqa: F811
    """Without tables the pass's first RX carries the last segment's factors."""
    n = 4
    circ = [G("RX", (q,), param=2.7) for _ in range(1200) for q in range(n)]
    got, _ = emulator(n, circ, mode="tile", dtype=dtype, arith=arith, tile_bits=n, fuse=False)
    check(got, circ, n)
    assert emulator.max_register_abs < 2.0 ** 25, emulator.max_register_abs
    least = 2.0 ** -25 * (min_cos(circ) if arith == "df" else 1.0)
    assert emulator.min_register_scale > least, (emulator.min_register_scale, least)
