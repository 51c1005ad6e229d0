"""The programs the tile kernels run -- lowered register ops (tables and phases on one or two slots, groups of
phases) and passes packed into kernel parameters -- executed on the host against the oracle (no GPU).

`plan_lowering_host.cpp` runs the library's own lowering.  A wrong slot, reordering, group or re-based entry
gives an O(1) error; the emulation's rounding is ~1e-15 and a double-float entry keeps 2^-48 relative
(a few thousand of them: 1e-11), so the bound is 1e-10."""
import os
import struct
import subprocess

import numpy as np
import pytest
from test_gpu_regops import circuit as slot_circuit
from test_gpu_tile_programs import circuits as program_circuits
from test_plan_emulator_host import CSRC, HERE, TOL, _lib, _nvcc, qs

from oracle import sv
from workloads import circuits as wc


@pytest.fixture(scope="module")
def lowered(tmp_path_factory):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("lowering")
    exe = str(d / "plan_lowering_host")
    srcs = [os.path.join(HERE, "plan_lowering_host.cpp")] + \
        [os.path.join(CSRC, f) for f in ("gates.cpp", "compiler.cpp", "stages.cpp", "lowering.cpp")]
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-o", exe] + srcs, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]

    def run(n, circ, sms=152, **opts):
        """Checks both executions against the oracle; returns the counts of passes, programs and op kinds."""
        ops, nops, mats = qs.marshal(circ)
        inp, out = str(d / "in.bin"), str(d / "out.bin")
        with open(inp, "wb") as f:
            f.write(struct.pack("<iiq", n, nops, mats.size) + bytes(qs._opts(mode="tile", **opts)) + struct.pack("<i", 0))
            f.write(bytes(_lib.qs_cost_model()) + bytes(ops)[: nops * 48])
            f.write(np.ascontiguousarray(mats, dtype=np.float64).tobytes())
        r = subprocess.run([exe, inp, out, str(sms)], capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, (r.returncode, r.stderr[-3000:])
        with open(out, "rb") as f:
            f.read(4)
            sigma = np.frombuffer(f.read(4 * n), dtype=np.int32)
            states = np.frombuffer(f.read(), dtype=np.complex128).reshape(2, -1)
        ar = np.arange(1 << n, dtype=np.int64)
        idx = sum(((ar >> q) & 1) << int(sigma[q]) for q in range(n))
        ref = sv.simulate(n, circ)
        for s in states:
            assert np.max(np.abs(s[idx] - ref)) <= TOL
        w = r.stderr.split()
        return {w[i]: int(w[i + 1]) for i in range(0, len(w), 2)}

    return run


@pytest.mark.parametrize("dtype,arith,K", [("c64", "auto", k) for k in (1, 2, 3, 4, 5)] +
                         [("c128", a, k) for a in ("df", "f64") for k in (1, 2, 3, 4)])
@pytest.mark.parametrize("n,tile,phases", [(5, 5, 1), (10, 6, 2), (11, 8, 8)])
def test_factors_on_few_slots(lowered, dtype, arith, K, n, tile, phases):
    got = lowered(n, slot_circuit(n, 100 * n + K, min(phases, n - 2)), dtype=dtype, arith=arith, tile_bits=tile, reg_bits=K)
    assert n == 5 or got["slot"] + got["dtab2"] + got["grouped"] > 0
    assert got["grouped"] == 0 or arith == "df"


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,tile", [(6, 0), (9, 0), (12, 0), (12, 8), (13, 9)])
def test_programs(lowered, dtype, n, tile):
    """The circuits of the kernels' own test, from one pass for the whole circuit to passes of a few stages; no
    double-float pass has a program where it has more tiles than SMs."""
    kw = {"dtype": dtype, "tile_bits": tile, "dense": False}
    seen = {}
    for i, circ in enumerate(program_circuits(n, n)):
        got = lowered(n, circ, **kw)
        for k, v in got.items():
            seen[k] = seen.get(k, 0) + v
        if tile:   # passes short enough for the parameter space; 2: with SWAPs, 7: with dense blocks
            assert i in (2, 7) or got["programs"] == got["passes"], (i, got)
            assert i != 7 or got["programs"] == 0
        few = lowered(n, circ, sms=0, **kw)
        assert few["programs"] == (0 if dtype == "c128" else got["programs"])
    assert seen["programs"] > 0 and seen["dtab2"] > 0 and seen["slot"] > 0
    assert (seen["grouped"] > 0) == (dtype == "c128")


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_programs_of_refused_forms(lowered, dtype):
    n = 9
    long = wc.haar_cnot_circuit(n, 160, 1)
    assert lowered(n, long, dtype=dtype)["programs"] == 0
    dense = [wc.Gate("H", (q,)) for q in range(n)] + [wc.Gate("U2", (0, 5), matrix=wc.haar_unitary(4, np.random.default_rng(1)))]
    assert lowered(n, dense, dtype=dtype, dense=False)["programs"] == 0
    short = wc.rzrx_cz_circuit(n, 4, 1)
    assert lowered(n, short, dtype=dtype)["programs"] > 0
    assert lowered(n, short, dtype=dtype, reg_bits=3)["programs"] == 0
    if dtype == "c128":
        assert lowered(n, short, dtype=dtype, arith="f64")["programs"] == 0
        assert lowered(n, short, dtype=dtype, tile_bits=6, sms=8)["programs"] > 0
        assert lowered(n, short, dtype=dtype, tile_bits=6, sms=7)["programs"] == 0
