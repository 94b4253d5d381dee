"""FP32 k = 5, 6 operators against the oracle at the edges of the tile kernel:
one tile, two (one per team), an odd number per CTA, and target placements with
and without position 0, packed low, spread and high, in unsorted order.  Sums of
at most 64 FP32 terms stay far below the suite's 1e-5."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_helpers import GState, check_close  # noqa: E402


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_16940_gb300 as q
    return q


@pytest.mark.parametrize("n", [11, 12, 13, 16, 21])
@pytest.mark.parametrize("k", [5, 6])
def test_wide_fp32_placements(q, n, k):
    rng = np.random.default_rng(10 * n + k)
    sets = [list(range(k)), list(range(n - k, n)), [0] + list(range(n - k + 1, n)), [0, 1, 3, 5, 8, 10][:k],
            [1, 2, 3, 4, n - 1, 6][:k], [0, 2, 4, 6, 8, 10][:k]]
    psi = W.random_state(n, seed=n).astype(np.complex64)
    want = psi.astype(np.complex128)
    st = GState(q, torch, n, init=psi)
    try:
        for s in sets:
            t = [int(v) for v in rng.permutation(s)]
            U = W.haar_unitary(1 << k, rng)
            q.qsa_apply_fused(st.h, t, U)
            oracle.apply(want, t, U)
            check_close(want, st.logical())
    finally:
        st.close()
