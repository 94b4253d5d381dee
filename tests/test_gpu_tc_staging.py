"""Output staging of the tensor-core pass: with no target at position 0 the
fourth target decides whether 16-byte units are staged with their halves
swapped.  It goes through every chunk-local position it can have: a bit of the
lane's unit (4, 5) or of the unit number (6 and above), for one chunk, for the
half-filled last pair of an odd chunk count, and beside targets 1..3 and above.
Bounds: those of the single-operator tests (FP64 oracle)."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import GState, check_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [11, 12, 19])
@pytest.mark.parametrize("p", [4, 5, 6, 7, 8, 9, 10])
def test_swapped_halves_read_back(p, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_16940_gb300 as q
    rng = np.random.default_rng(16 * n + p)
    psi = W.random_state(n, seed=n)
    st = GState(q, torch, n, init=psi.astype(np.complex64))
    ref = psi.astype(np.complex64).astype(np.complex128)
    try:
        sets = [(1, 2, 3, p, n - 1), (3, p - 1, 1, n - 1, p, n - 2)]
        for t in sets:
            t = tuple(dict.fromkeys(t))
            if len(t) < 5:
                continue
            G = W.haar_unitary(1 << len(t), rng)
            q.qsa_apply_fused_ex(st.h, t, G, q.QSA_LOWER_STRIDED, q.QSA_PREC_TF32X3)
            oracle.apply(ref, t, G)
        check_close(ref, st.logical())
    finally:
        st.close()
