"""Outcomes of many shots within their blocks of 1024 amplitudes, bit for bit
against the oracle: the weight at one or two places of a block's search (first
and last amplitude, both sides of a pair and of a run of 16 pairs), with zeros
between, and components of magnitude 2, whose weights take the wider form."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_helpers import GState  # noqa: E402


@pytest.mark.parametrize("value", [0.5, 2.0, -2.0j])
@pytest.mark.parametrize("places", [(0,), (1023,), (31, 32), (30, 33), (511, 512), (1022, 1024)])
def test_places_within_a_block(places, value):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_16940_gb300 as q
    n, shots = 13, 6000
    psi = W.random_state(n, seed=3, zero_frac=0.5).astype(np.complex64)
    psi[2048:4096] = 0
    for p in places:
        psi[2048 + p] = value
    st = GState(q, torch, n, init=psi)
    try:
        want_v, want_c = oracle.sample_counts(psi.astype(np.complex128), list(range(n)), shots, 5)
        v, c = q.qsa_sample_counts(st.h, shots, seed=5)
        assert np.array_equal(v, want_v) and np.array_equal(c, want_c)
    finally:
        st.close()
