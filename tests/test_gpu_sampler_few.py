"""Up to 4096 shots (sorted and run-length encoded by one CTA, a warp a shot) bit
for bit against the oracle: shot counts around the powers of two and of 32, where
the keys of a thread and the padding change, states below one block of 1024
amplitudes, of one block and of many (the block search's steps of 32), permuted
layouts, and outcomes that repeat.  One state of 33 qubits takes 64-bit keys."""
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


@pytest.mark.parametrize("n", [3, 9, 10, 11, 15, 16, 21])
def test_few_shots_match_oracle(q, n):
    rng = np.random.default_rng(n)
    psi = W.random_state(n, seed=n, zero_frac=0.3).astype(np.complex64)
    L = [int(v) for v in rng.permutation(n)]
    x = np.arange(1 << n)
    y = np.zeros_like(x)
    for j in range(n):
        y |= ((x >> j) & 1) << L[j]
    stored = np.zeros_like(psi)
    stored[y] = psi
    st = GState(q, torch, n)
    try:
        q.qsa_set_layout(st.h, L, materialise=0)
        st.buf.copy_(torch.from_numpy(stored))
        for shots in (1, 2, 31, 33, 64, 100, 1023, 1024, 1025, 2047, 2049, 4095, 4096):
            want_v, want_c = oracle.sample_counts(psi.astype(np.complex128), L, shots, shots)
            v, c = q.qsa_sample_counts(st.h, shots, seed=shots)
            assert np.array_equal(v, want_v) and np.array_equal(c, want_c)
    finally:
        st.close()


def test_wide_keys(q):
    n = 33
    if torch.cuda.mem_get_info()[0] < 80 << 30:
        pytest.skip("needs 80 GB")
    buf = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
    at = [0, 5, (1 << 32) - 1, 1 << 32, (1 << 33) - 1]
    for i in at:
        buf[i] = 5 ** -0.5
    h = q.qsa_state_create_ex(n, buf.data_ptr(), buf.numel() * 8, torch.cuda.current_stream().cuda_stream, 0)
    try:
        for shots in (1000, 2000, 4096):
            v, c = q.qsa_sample_counts(h, shots, seed=1)
            assert v.tolist() == at and int(c.sum()) == shots
            # five equal outcomes: each count within 6 standard deviations
            assert np.all(np.abs(c.astype(np.float64) - shots / 5) < 6 * np.sqrt(shots * 0.16))
    finally:
        q.qsa_state_destroy(h)
        del buf
        torch.cuda.empty_cache()
