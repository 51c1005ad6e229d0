"""GPU: long passes whose RX angles all lie near pi, single plan and batch, against the FP64 oracle, at the
complex128 tolerance of 1e-12 per amplitude.  4800 rotations add about 2^-48 of rounding each (2.5e-13 of
the norm as a random walk).  What equal angles add up coherently is larger where low parts grow through the
whole pass (1.4e-12 here); the RX that close the tangent segments normalise them."""
import numpy as np
import pytest
from test_tangent_segments_host import kicked_chain

from oracle import sv

pytestmark = pytest.mark.gpu

qs = pytest.importorskip("paper_2010_09746_gb300")


@pytest.mark.parametrize("angle", [0.85 * np.pi, (0.85 * np.pi, 1.15 * np.pi)], ids=["fixed", "drawn"])
@pytest.mark.parametrize("arith", ["df", "f64"])
def test_angles_near_pi(arith, angle):
    n = 12
    circ = kicked_chain(n, 400, angle)
    ref = sv.simulate(n, circ)
    st = qs.State(n, "c128", arith=arith)
    st.execute(qs.compile(n, circ, mode="tile", dtype="c128", arith=arith))
    assert np.abs(st.amplitudes() - ref).max() <= 1e-12
    assert abs(st.norm() - 1.0) <= 1e-11
    if arith == "df":
        b = qs.Batch([(n, circ), (n, circ[: len(circ) // 2])], dtype="c128")
        b.run()
        assert np.abs(b.amplitudes(0) - ref).max() <= 1e-12
        assert np.abs(b.amplitudes(1) - sv.simulate(n, circ[: len(circ) // 2])).max() <= 1e-12
