"""Layout changes and bit swaps, bit for bit: random permutations of all
positions (long cycles cut over several passes), single cycles, reversals and
identities, on states smaller than, equal to and larger than a pass's tile of
2^13 amplitudes."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_helpers import GState  # noqa: E402


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_16940_gb300 as q
    return q


def _stored(psi, n, L):
    """Logical vector in stored order: bit L[j] of the index is logical bit j."""
    x = np.arange(1 << n)
    y = np.zeros_like(x)
    for j in range(n):
        y |= ((x >> j) & 1) << L[j]
    out = np.empty_like(psi)
    out[y] = psi
    return out


@pytest.mark.parametrize("n", [2, 4, 9, 12, 13, 14, 17, 22])
def test_layouts_and_swaps_bit_exact(q, n):
    rng = np.random.default_rng(n)
    psi = W.random_state(n, seed=n).astype(np.complex64)
    st = GState(q, torch, n, init=psi)
    try:
        L = list(range(n))
        layouts = [rng.permutation(n).tolist() for _ in range(4)]
        layouts += [[(j + 1) % n for j in range(n)], [n - 1 - j for j in range(n)], list(range(n)), list(range(n))]
        for lay in layouts:
            q.qsa_set_layout(st.h, lay)
            L = lay
            assert q.qsa_get_layout(st.h) == L
            torch.cuda.synchronize()
            assert np.array_equal(st.buf.cpu().numpy(), _stored(psi, n, L))
            p = rng.permutation(n)
            k = n // 2
            a, b = p[:k].tolist(), p[k:2 * k].tolist()
            q.qsa_permute_bits(st.h, a, b)
            swap = dict(zip(a + b, b + a))
            L = [swap.get(x, x) for x in L]
            assert q.qsa_get_layout(st.h) == L
            torch.cuda.synchronize()
            assert np.array_equal(st.buf.cpu().numpy(), _stored(psi, n, L))
    finally:
        st.close()
