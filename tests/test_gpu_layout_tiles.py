"""Bit swaps whose number of high positions lies around the line between the two
tile sizes of a permutation pass (nine positions above the lowest three) and
around the line to a second pass (ten), on states at and around one tile and on
both sides of the L2, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_helpers import GState  # noqa: E402


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_16940_gb300 as q
    return q


@pytest.mark.parametrize("n,pairs,low", [(n, p, low) for n in (12, 13, 14, 15, 23, 24)
                                         for p, low in ((1, 0), (1, 1), (4, 0), (5, 1), (5, 0), (6, 2), (6, 1), (6, 0))
                                         if 2 * p - low + 3 <= n])
def test_swaps_around_the_tile_sizes(q, n, pairs, low):
    """pairs swaps, low of them of one of the three lowest positions."""
    rng = np.random.default_rng(100 * n + 10 * pairs + low)
    lows = rng.permutation(3)[:low].tolist()
    highs = (3 + rng.permutation(n - 3)[:2 * pairs - low]).tolist()
    a, b = lows + highs[:pairs - low], highs[pairs - low:]
    st = GState(q, torch, n)
    try:
        x = torch.arange(1 << n, device="cuda")
        st.buf.copy_(torch.complex(x.float(), -x.float()))   # integers below 2^24: exact
        q.qsa_permute_bits(st.h, a, b)
        y = x.clone()
        for p, r in zip(a, b):
            d = ((x >> p) ^ (x >> r)) & 1
            y ^= (d << p) | (d << r)
        torch.cuda.synchronize()
        assert torch.equal(st.buf, torch.complex(y.float(), -y.float()))
    finally:
        st.close()
