"""Samplers with many shots (radix-sorted outcomes, shots grouped by block)
bit for bit against the oracle: shot counts around the tile of 1024 keys and the
4096-key limit of the one-CTA sort, states of one block and of many, more and
fewer shots than blocks, permuted layouts, a state with empty bins, and
outcomes that repeat often (a few large amplitudes)."""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("n,shots,kind", [(6, 5000, "random"), (9, 6145, "zeros"), (10, 4097, "random"),
                                          (11, 8192, "peaked"), (14, 70001, "random"), (17, 20000, "zeros"),
                                          (20, 5000, "peaked"), (22, 4500, "random"), (24, 4097, "random")])
def test_many_shots_match_oracle(q, n, shots, kind):
    rng = np.random.default_rng(n + shots)
    psi = W.random_state(n, seed=n, zero_frac=0.6 if kind == "zeros" else 0.0).astype(np.complex64)
    if kind == "peaked":
        psi *= 1e-3
        psi[rng.integers(0, 1 << n, 5)] = 0.44
    L = [int(v) for v in rng.permutation(n)]
    st = GState(q, torch, n)
    try:
        q.qsa_set_layout(st.h, L, materialise=0)
        stored = np.zeros_like(psi)   # stored order: logical x at y, bit L[j] of y = bit j of x
        x = np.arange(1 << n)
        y = np.zeros_like(x)
        for j in range(n):
            y |= ((x >> j) & 1) << L[j]
        stored[y] = psi
        st.buf.copy_(torch.from_numpy(stored))
        want_v, want_c = oracle.sample_counts(psi.astype(np.complex128), L, shots, 99)
        for _ in range(2):
            v, c = q.qsa_sample_counts(st.h, shots, seed=99)
            assert np.array_equal(v, want_v) and np.array_equal(c, want_c)
            assert int(c.sum()) == shots
    finally:
        st.close()
