"""<Z_mask> sums taken in the sampler's pass: one to four masks without and with
the qubit on the lowest position (its two amplitudes enter with the same or with
opposite signs), against FP64 numpy sums.  Bound: a thread's double-float sum
keeps about 48 bits, threads are combined in FP64, so 1e-12 on sums below 1."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_helpers import GState  # noqa: E402


@pytest.mark.parametrize("n", [10, 13, 18])
@pytest.mark.parametrize("count", [1, 2, 3, 4])
@pytest.mark.parametrize("low", [False, True])
def test_masks_with_and_without_the_lowest_position(n, count, low):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_16940_gb300 as q
    rng = np.random.default_rng(8 * n + count)
    psi = W.random_state(n, seed=n).astype(np.complex64)
    masks = [0] + [int(rng.integers(1, 1 << n)) & ~1 for _ in range(count - 1)]
    if low:
        masks[-1] |= 1
    st = GState(q, torch, n, init=psi)
    try:
        z, _, c = q.qsa_measure(st.h, masks, 200, 7)
        p = psi.real.astype(np.float64) ** 2 + psi.imag.astype(np.float64) ** 2
        x = np.arange(1 << n)
        for m, got in zip(masks, z):
            sign = 1 - 2 * (np.array([bin(v).count("1") for v in (x & m)]) & 1)
            assert abs(got - float((sign * p).sum())) < 1e-12
        assert int(c.sum()) == 200
    finally:
        st.close()
