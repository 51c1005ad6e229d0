"""Complex64 passes without moves (RZ / RX / CZ) leave the kernel parameters from 2^14 tiles on; passes with
moves stay there, and the lowered programs give the oracle's state either way (no GPU)."""
import pytest
from test_plan_lowering_host import lowered  # noqa: F401  (the fixture)

from workloads import circuits as wc


@pytest.mark.parametrize("n,light_programs", [(18, True), (19, False)])
def test_line_between_the_kernels(lowered, n, light_programs):  # noqa: F811
    tile = 5   # 2^13 and 2^14 tiles
    light = [wc.Gate(k, (q,), param=0.3 + q) for q in range(4) for k in ("RZ", "RX")] + [wc.Gate("CZ", (0, 3))]
    got = lowered(n, light, dtype="c64", tile_bits=tile, low_bits=2)
    assert got["passes"] > 0 and got["programs"] == (got["passes"] if light_programs else 0)
    moves = light + [wc.Gate("CNOT", (0, 1)), wc.Gate("RX", (1,), param=0.5)]
    got = lowered(n, moves, dtype="c64", tile_bits=tile, low_bits=2)
    assert got["passes"] > 0 and got["programs"] == got["passes"]
