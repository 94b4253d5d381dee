"""How an operator's products are added, by its error against 64 bits.

An output of a dense operator on D = 2^k amplitudes is a sum of 2 D products
per component.  With rounding errors of relative size d (2^-24 / sqrt(3) over a
mantissa spread evenly in logarithm: d = 2.53e-8) and terms of equal variance,
the sums of the D products of real and of the D products of imaginary parts,
added at the end, have the relative error d sqrt((D + 1) / 2 + 2), with the
rounding of the matrix and of the last addition; one running sum over all 2 D
products d sqrt((2 D + 1) / 2 + 1), 1.10, 1.21 and 1.35 times as much at k = 2, 3
and 5.  The bounds below lie at 1.05 times the first."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_helpers import GState  # noqa: E402

D_ROUND = 2.0 ** -24 * np.sqrt(0.375 / np.log(2.0) / 3.0)


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_16940_gb300 as q
    return q


def _relative_error(q, n, ops, opts, seed):
    psi = W.random_state(n, seed=seed).astype(np.complex64)
    want = psi.astype(np.complex128)
    for o in ops:
        oracle.apply(want, o.targets, o.matrix)
    st = GState(q, torch, n, init=psi)
    try:
        stats = q.qsa_apply_circuit(st.h, ops, opts)
        return np.linalg.norm(st.logical() - want) / np.linalg.norm(want), stats
    finally:
        st.close()


def _mean_error(q, n, k, count, opts):
    errs = []
    for seed in range(6):
        rng = np.random.default_rng(100 * k + seed)
        ops = [W.Op(tuple(int(t) for t in rng.permutation(n)[:k]), W.haar_unitary(1 << k, rng), False, "u")
               for _ in range(count)]
        e, stats = _relative_error(q, n, ops, opts, seed)
        errs.append(e)
    return np.sqrt(np.mean(np.square(errs))), stats


def _bound(k, count):
    return 1.05 * D_ROUND * np.sqrt(((1 << k) + 1) / 2 + 2) * np.sqrt(count)


def test_five_qubit_operators(q):
    e, _ = _mean_error(q, 14, 5, 4, q.make_opts(planner=q.QSA_PLAN_PER_GATE, kmax=5))
    assert e <= _bound(5, 4)


@pytest.mark.parametrize("k", [2, 3])
def test_grouped_operators(q, k):
    """Twelve operators, several to a pass."""
    e, stats = _mean_error(q, 14, k, 12, q.make_opts(planner=q.QSA_PLAN_GREEDY, kmax=k))
    assert stats["blocks"] == 12 and stats["passes"] < 12
    assert e <= _bound(k, 12)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 7, 9, 11])
def test_large_products(q, k):
    """N = 24, where some products run as layers: no further from 64 bits than the
    complex butterflies, whose factors have sums of four products each (relative
    error d sqrt(3.5) a factor; a tenth more for the spread over the factors drawn)."""
    n, errs = 24, []
    for seed in range(8):
        rng = np.random.default_rng(1000 * k + seed)
        t = [int(v) for v in rng.permutation(n)[:k]]
        fac = [W.haar_unitary(2, rng) for _ in range(k)]
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.view_as_complex(torch.randn(1 << n, 2, device="cuda", generator=g)) / 2 ** 12.5
        want = x.to(torch.complex128)
        for p, f in zip(t, fac):
            m = torch.from_numpy(np.ascontiguousarray(f)).cuda()
            want = torch.einsum("rc,acb->arb", m, want.view(-1, 2, 1 << p)).reshape(-1)
        st = GState(q, torch, n)
        try:
            st.buf.copy_(x)
            q.qsa_apply_product(st.h, t, fac)
            d = torch.linalg.vector_norm(st.buf.to(torch.complex128) - want)
            errs.append(float(d / torch.linalg.vector_norm(want)))
        finally:
            st.close()
    assert np.sqrt(np.mean(np.square(errs))) <= 1.1 * D_ROUND * np.sqrt(3.5 * k)


@pytest.mark.parametrize("n", [13, 20])
def test_two_grouped_one_qubit_operators(q, n):
    """The shortest group: its phases and rotations cost no more than the two
    operators as complex 2 x 2 passes (sums of two and two products, relative error
    d sqrt(3.5) each; a tenth more for the spread over the operators drawn)."""
    errs = []
    for seed in range(12):
        rng = np.random.default_rng(seed)
        ops = [W.Op((t,), W.haar_unitary(2, rng), False, "u") for t in (3, 7)]
        e, stats = _relative_error(q, n, ops, q.make_opts(planner=q.QSA_PLAN_GREEDY, kmax=1), seed)
        assert stats["blocks"] == 2 and stats["passes"] == 1
        errs.append(e)
    assert np.sqrt(np.mean(np.square(errs))) <= 1.1 * D_ROUND * np.sqrt(3.5 * 2)


@pytest.mark.parametrize("n", [23, 24])
def test_three_qubit_operators_in_and_beyond_the_l2(q, n):
    """Packed and scalar FMAs, both with two sums: the same bound."""
    errs = []
    for seed in range(4):
        rng = np.random.default_rng(seed)
        t = sorted(int(v) for v in rng.permutation(n)[:3])
        m = W.haar_unitary(8, rng)
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.view_as_complex(torch.randn(1 << n, 2, device="cuda", generator=g)) / 2 ** 12
        # axes: bits above t[2], t[2], between, t[1], between, t[0], below
        v = x.to(torch.complex128).view(1 << (n - 1 - t[2]), 2, 1 << (t[2] - t[1] - 1), 2, 1 << (t[1] - t[0] - 1), 2,
                                        1 << t[0])
        want = torch.einsum("cbafed,ufvewdx->ucvbwax", torch.from_numpy(m.reshape([2] * 6)).cuda(), v).reshape(-1)
        st = GState(q, torch, n)
        try:
            st.buf.copy_(x)
            q.qsa_apply_fused(st.h, t, m)
            d = torch.linalg.vector_norm(st.buf.to(torch.complex128) - want)
            errs.append(float(d / torch.linalg.vector_norm(want)))
        finally:
            st.close()
    assert np.sqrt(np.mean(np.square(errs))) <= _bound(3, 1)
