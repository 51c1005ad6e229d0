"""GPU: the permutation kernel where its tiles change shape: states smaller than a tile, low bits that
stay, move among themselves or go to the top, bit 0 fixed (complex64 pairs) or not, and every bit
moved; bit for bit against the definition."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

qs = pytest.importorskip("paper_2010_09746_gb300")


def perms(n, rng):
    ident = list(range(n))
    yield ident[::-1]                              # every low bit to the top
    yield ident[1:] + ident[:1]                    # rotation by one
    yield [int(x) for x in rng.permutation(n)]
    p = list(ident)                                # one exchange that keeps bit 0
    p[n - 1], p[n // 2] = p[n // 2], p[n - 1]
    yield p
    p = [0] + [1 + int(x) for x in rng.permutation(n - 1)]   # bit 0 fixed, the rest shuffled
    yield p


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", [2, 3, 5, 8, 9, 10, 11, 12, 13, 16, 21])
def test_permutations(dtype, n):
    rng = np.random.default_rng(n)
    st = qs.State(n, dtype)
    N = 1 << n
    ref = (np.arange(N) + 1j * (N - np.arange(N))).astype(st.np_dtype)   # every amplitude distinct
    st.set_amplitudes(ref)
    i = np.arange(N)
    for p in perms(n, rng):
        st.permute(p)
        j = np.zeros(N, dtype=np.int64)
        for q in range(n):
            j |= ((i >> q) & 1) << p[q]
        want = np.empty_like(ref)
        want[j] = ref
        assert st.amplitudes(order=qs.QS_ORDER_STORAGE).tobytes() == want.tobytes(), p
