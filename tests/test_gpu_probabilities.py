"""Probabilities in logical order, bit for bit against numpy's FP64 squares
(fl64(re^2) + fl64(im^2)): sizes below, at and above one tile of 2^12
amplitudes, random layouts, amplitudes that are zero, subnormal, huge, infinite
or NaN, and an output that starts off a 16-byte boundary."""
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


@pytest.mark.parametrize("n", [1, 5, 11, 12, 13, 15, 19])
@pytest.mark.parametrize("special", [False, True])
@pytest.mark.parametrize("shift", [0, 1])
def test_probabilities_bit_exact(q, n, special, shift):
    rng = np.random.default_rng(n)
    L = [int(v) for v in rng.permutation(n)]
    psi = W.random_state(n, seed=n).astype(np.complex64)   # stored order
    if special:
        f = psi.view(np.float32)
        pick = rng.integers(0, 8, f.size)
        for i, v in enumerate([0.0, 1e-42, -3e-39, 1.1754944e-38, 2e30, np.inf, np.nan]):
            f[pick == i] = v
    st = GState(q, torch, n)
    try:
        q.qsa_set_layout(st.h, L, materialise=0)
        st.buf.copy_(torch.from_numpy(psi))
        out = torch.full(((1 << n) + 2,), -1.0, dtype=torch.float64, device="cuda:0")
        norm = q.qsa_probabilities_device(st.h, out.data_ptr() + 8 * shift)
        got = out.cpu().numpy()
        x = np.arange(1 << n)
        y = np.zeros_like(x)
        for j in range(n):
            y |= ((x >> j) & 1) << L[j]
        with np.errstate(all="ignore"):
            want = psi.real.astype(np.float64) ** 2 + psi.imag.astype(np.float64) ** 2
        assert np.array_equal(got[shift:shift + (1 << n)], want[y], equal_nan=True)
        assert np.all(np.delete(got, np.s_[shift:shift + (1 << n)]) == -1.0)   # nothing written around it
        if not special:
            assert abs(norm - want.sum()) < 1e-12   # about 48 bits per thread's partial sum, FP64 across threads
            assert abs(q.qsa_expectation_z(st.h, 0) - norm) < 1e-12
    finally:
        st.close()
