"""Products on states large enough for the layer path, against each other: the
product of unitary factors (a layer) on some qubits, then the inverse product
scaled by 2 and 1/2 (not unitary: the product kernel's complex butterflies)
returns the state; the first also against the one-qubit kernel, factor by
factor.  FP32 errors of 1 + 11 passes stay far below 1e-5 of the largest
amplitude's scale."""
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


@pytest.mark.parametrize("k", [1, 2, 7, 11])
@pytest.mark.parametrize("high", [False, True])
def test_large_products(q, k, high):
    n = 24
    rng = np.random.default_rng(k)
    t = [int(v) for v in (rng.permutation(np.arange(n - k, n)) if high else rng.permutation(n)[:k])]
    fac = [W.haar_unitary(2, rng) for _ in range(k)]
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.view_as_complex(torch.randn(1 << n, 2, device="cuda", generator=g))
    sts = [GState(q, torch, n) for _ in range(2)]
    try:
        for s in sts:
            s.buf.copy_(x)
        q.qsa_apply_product(sts[0].h, t, fac)
        for j in range(k):
            q.qsa_apply_fused(sts[1].h, [t[j]], fac[j])
        torch.cuda.synchronize()
        assert float((sts[0].buf - sts[1].buf).abs().max()) <= 1e-5 * float(x.abs().max())
        inv = [f.conj().T * (2.0 if j % 2 else 0.5) for j, f in enumerate(fac)]
        q.qsa_apply_product(sts[0].h, t, inv)
        torch.cuda.synchronize()
        scale = float(np.prod([2.0 if j % 2 else 0.5 for j in range(k)]))
        assert float((sts[0].buf / scale - x).abs().max()) <= 1e-5 * float(x.abs().max())
    finally:
        for s in sts:
            s.close()
