"""Group passes at the edges of what they accept: groups that multiply to the
identity and so have no pass, factors with entries that are not numbers (those
also where products run as layers), allocations that fail before the first pass,
what a plan uploads for grouped products, programs longer than a pass holds, the
largest grouped state, and operators that are not unitary.  Same tolerance as the
other group tests (1e-5 on fidelity and amplitudes, FP32 sums of at most 32 terms
over a few blocks)."""
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


def _identity_then(n, tail, rng):
    """Identities on every qubit; "dense": then a dense k = 5 block, which no
    group takes, and one-qubit unitaries."""
    ops = [W.Op((j,), np.eye(2), False, "i") for j in range(n)]
    if tail == "dense":
        ops.append(W.Op(tuple(int(t) for t in rng.permutation(n)[:5]), W.haar_unitary(32, rng), False, "u"))
        ops += [W.Op((j,), W.haar_unitary(2, rng), False, "u") for j in range(n)]
    return ops


@pytest.mark.parametrize("n", [5, 12, 14])
@pytest.mark.parametrize("tail", ["none", "dense"])
def test_identity_group_from_zero(q, n, tail):
    """Run from |0...0> on a buffer that holds something else."""
    rng = np.random.default_rng(n)
    ops = _identity_then(n, tail, rng)
    L = [int(v) for v in rng.permutation(n)]
    plan = q.qsa_plan_create(ops, n, q.make_opts(planner=q.QSA_PLAN_DP, kmax=1), layout=L)
    st = GState(q, torch, n, init=W.random_state(n, seed=n).astype(np.complex64))
    try:
        stats = q.qsa_plan_execute_from_zero(st.h, plan)
        assert stats["blocks"] == len(ops) and q.qsa_get_layout(st.h) == L
        check_close(oracle.run_circuit(n, ops), st.logical())
        # operators were applied, so |0...0> is no longer taken for granted
        with pytest.raises(q.QsaError):
            q.qsa_set_layout(st.h, list(range(n)), materialise=0)
    finally:
        st.close()
        q.qsa_plan_destroy(plan)


def test_identity_trajectory(q):
    """A batch whose trajectories are empty after that: |0...0> itself."""
    n, rng = 6, np.random.default_rng(6)
    trajs = [_identity_then(n, "none", rng), [], [W.Op((2,), W.X, False, "x")]]
    b = q.qsa_batch_create(n, trajs, q.make_opts(planner=q.QSA_PLAN_DP, kmax=1, kmax_diag=1))
    x = torch.randn(3, 1 << n, dtype=torch.complex64, device="cuda:0")
    try:
        q.qsa_batch_run(b, x.data_ptr(), x.numel() * 8, 10, 1)
        for got, ops in zip(x.cpu().numpy().astype(np.complex128), trajs):
            check_close(oracle.run_circuit(n, ops), got)
    finally:
        q.qsa_batch_destroy(b)


BAD = [(i, v) for i in range(4) for v in (np.nan, complex(0, np.nan))]


def _with_bad(i, v, rng):
    F = W.haar_unitary(2, rng) if i != 2 else np.diag([1.0, 1.0]).astype(np.complex128)
    F.flat[i] = v
    return F


def _check_bad(ops, psi, got):
    """Wherever the oracle's amplitude is not a number, neither is the library's."""
    want = psi.astype(np.complex128)
    with np.errstate(invalid="ignore"):
        for o in ops:
            oracle.apply(want, o.targets, o.matrix)
    assert np.isnan(want).any()
    assert np.isnan(got[np.isnan(want)]).all()


@pytest.mark.parametrize("i,v", BAD)
@pytest.mark.parametrize("n", [5, 13])
@pytest.mark.parametrize("kind", ["one-qubit blocks", "product blocks", "layer"])
def test_not_a_number_in_a_plan(q, n, kind, i, v):
    rng = np.random.default_rng(10 * n + i)
    ops = [W.Op((j,), W.haar_unitary(2, rng), False, "u") for j in range(n)]
    ops[3] = W.Op((3,), _with_bad(i, v, rng), False, "bad")
    opts = {"one-qubit blocks": dict(kmax=1), "product blocks": dict(kmax=1, kmax_prod=3),
            "layer": dict(kmax=4, layer=1)}[kind]
    psi = W.random_state(n, seed=i).astype(np.complex64)
    st = GState(q, torch, n, init=psi)
    try:
        q.qsa_apply_circuit(st.h, ops, q.make_opts(planner=q.QSA_PLAN_DP, **opts))
        _check_bad(ops, psi, st.logical())
    finally:
        st.close()


@pytest.mark.parametrize("i,v", BAD)
def test_not_a_number_in_a_batch(q, i, v):
    n, rng = 5, np.random.default_rng(i)
    ops = [W.Op((2,), W.haar_unitary(2, rng), False, "u"), W.Op((2,), _with_bad(i, v, rng), False, "bad"),
           W.Op((2,), W.haar_unitary(2, rng), False, "u")]
    b = q.qsa_batch_create(n, [ops], q.make_opts(planner=q.QSA_PLAN_DP, kmax=1, kmax_diag=1))
    x = torch.zeros(1 << n, dtype=torch.complex64, device="cuda:0")
    zero = np.zeros(1 << n, dtype=np.complex64)
    zero[0] = 1
    try:
        q.qsa_batch_run(b, x.data_ptr(), x.numel() * 8, 1, 1)
        _check_bad(ops, zero, x.cpu().numpy().astype(np.complex128))
    finally:
        q.qsa_batch_destroy(b)


@pytest.mark.parametrize("i,v", BAD)
@pytest.mark.parametrize("layer", [False, True])
def test_not_a_number_in_a_large_product(q, layer, i, v):
    """N = 24, where unitary products run as layers: the amplitudes whose qubit
    selects the row of the entry (both rows of a state without zeros are read)."""
    n, t, rng = 24, [2, 23], np.random.default_rng(i)
    fac = [_with_bad(i, v, rng), W.haar_unitary(2, rng)]
    st = GState(q, torch, n)
    try:
        st.buf.fill_(1.0)
        if layer:
            q.qsa_apply_layer(st.h, [], t, fac)
        else:
            q.qsa_apply_product(st.h, t, fac)
        row = torch.isnan(st.buf.view(-1, 2, 4)[:, i >> 1])
        assert bool(row.all())
    finally:
        st.close()


@pytest.mark.parametrize("kind", ["group", "zero_init"])
def test_from_zero_after_a_failed_allocation(q, kind):
    """Every allocation of the call fails once, on a state that holds other
    amplitudes in another layout: the state is then |0...0> in the plan's layout,
    and the call works once memory is there."""
    n = 13
    rng = np.random.default_rng(3)
    if kind == "group":
        ops, opts = _identity_then(n, "dense", rng)[n + 1:], dict(planner=q.QSA_PLAN_DP, kmax=1)
    else:
        ops, _ = W.qaoa_circuit(n=14, p=1, seed=4)
        n, opts = 14, dict(planner=q.QSA_PLAN_DP, kmax=6, kmax_diag=12, layer=1, zero_init=1)
    L = [int(v) for v in rng.permutation(n)]
    failures = 0
    for nth in range(8):
        plan = q.qsa_plan_create(ops, n, q.make_opts(**opts), layout=L)
        st = GState(q, torch, n, init=W.random_state(n, seed=n).astype(np.complex64))
        q.qsa_debug_fail_alloc(nth)
        try:
            try:
                q.qsa_plan_execute_from_zero(st.h, plan)
                break
            except q.QsaError as e:
                assert e.code == q.QSA_E_NOMEM
            finally:
                q.qsa_debug_fail_alloc(-1)
            failures += 1
            assert q.qsa_get_layout(st.h) == L
            zero = np.zeros(1 << n, dtype=np.complex128)
            zero[0] = 1
            assert np.array_equal(st.logical(), zero)
            q.qsa_plan_execute_from_zero(st.h, plan)
            check_close(oracle.run_circuit(n, ops), st.logical())
        finally:
            st.close()
            q.qsa_plan_destroy(plan)
    assert failures >= 1


def test_grouped_products_upload_no_layers(q):
    """Product blocks of a run go into group passes: on a state large enough for
    products as layers the plan holds no layer tables for them, so its upload is
    the one of a state below that size (the same targets, so the same programs)."""
    rng = np.random.default_rng(8)
    ops = [W.Op((j,), W.haar_unitary(2, rng), False, "u") for j in range(14)]
    h2d = []
    for n in (23, 24):
        plan = q.qsa_plan_create(ops, n, q.make_opts(planner=q.QSA_PLAN_DP, kmax=1, kmax_prod=7))
        assert list(q.qsa_plan_block_kinds(plan)[0]) == [2, 2]
        st = GState(q, torch, n)
        try:
            h2d.append(q.qsa_plan_execute(st.h, plan)["h2d_bytes"])
        finally:
            st.close()
            q.qsa_plan_destroy(plan)
    assert h2d[0] == h2d[1] > 0


@pytest.mark.parametrize("n,k,count", [(4, 4, 40), (5, 4, 60), (12, 4, 60), (13, 4, 45), (12, 3, 200), (12, 1, 700)])
def test_long_programs(q, n, k, count):
    """More operators on one tile than a pass's program holds: several passes, each
    filled as far as it goes (the errors of so many operators stay below 1e-5)."""
    rng = np.random.default_rng(1000 * n + count)
    ops = [W.Op(tuple(int(t) for t in rng.permutation(n)[:k]), W.haar_unitary(1 << k, rng), False, "u")
           for _ in range(count)]
    psi = W.random_state(n, seed=n).astype(np.complex64)
    plan = q.qsa_plan_create(ops, n, q.make_opts(planner=q.QSA_PLAN_GREEDY, kmax=k if n > 4 else 1))
    st = GState(q, torch, n, init=psi)
    try:
        stats = q.qsa_plan_execute(st.h, plan)
        assert 1 < stats["passes"] < stats["blocks"]
        want = psi.astype(np.complex128)
        for o in ops:
            oracle.apply(want, o.targets, o.matrix)
        check_close(want, st.logical())
    finally:
        st.close()
        q.qsa_plan_destroy(plan)


@pytest.mark.parametrize("n", [25, 26])
def test_both_sides_of_the_size_limit(q, n):
    """The same plan options, grouped and a pass per block, against one pass per
    operator."""
    rng = np.random.default_rng(n)
    ops = []
    for i in range(24):
        k = 1 + i % 3
        t = tuple(int(v) for v in rng.permutation(n)[:k])
        ops.append(W.Op(t, np.diag(np.exp(1j * rng.uniform(0, 6, 1 << k))), True, "d") if i % 4 == 3 else
                   W.Op(t, W.haar_unitary(1 << k, rng), False, "u"))
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.view_as_complex(torch.randn(1 << n, 2, device="cuda", generator=g))
    x /= torch.linalg.vector_norm(x)
    sts = [GState(q, torch, n) for _ in range(2)]
    try:
        for st in sts:
            st.buf.copy_(x)
        stats = q.qsa_apply_circuit(sts[0].h, ops, q.make_opts(planner=q.QSA_PLAN_GREEDY, kmax=4))
        assert stats["passes"] < stats["blocks"] if n <= 25 else stats["passes"] == stats["blocks"]
        q.qsa_apply_circuit(sts[1].h, ops, q.make_opts(planner=q.QSA_PLAN_PER_GATE, kmax=4))
        torch.cuda.synchronize()
        assert float(torch.linalg.vector_norm(sts[0].buf - sts[1].buf)) <= 1e-5
    finally:
        for st in sts:
            st.close()


def _general_ops(n, rng):
    """Operators that are not unitary, of norm about one: scaled unitaries, rank-one
    and zero factors, projectors, triangular and random 2 x 2 ones between
    rotations, wider dense ones, and diagonals of up to eight qubits with zeros and
    entries of very different size."""
    def pick(k):
        return tuple(int(v) for v in rng.permutation(n)[:k])
    ops = []
    for i in range(10):
        q0 = pick(1)
        ops.append(W.Op(q0, W.haar_unitary(2, rng), False, "u"))
        kind = i % 5
        if kind == 0:
            m = W.haar_unitary(2, rng) * (1.25 if i < 5 else 0.8)
        elif kind == 1:
            m = np.outer([0.6, 0.8j], [1.0, 1j])           # rank one
        elif kind == 2:
            m = np.diag([1.0, 0.0]).astype(np.complex128)  # a projector
        elif kind == 3:
            m = np.array([[0.9, 0.7], [0.0, 1.1]], dtype=np.complex128)
        else:
            m = 0.7 * (rng.standard_normal((2, 2)) + 1j * rng.standard_normal((2, 2)))
        ops.append(W.Op(q0 if i % 2 else pick(1), m, False, "m"))
        ops.append(W.Op(q0, W.haar_unitary(2, rng), False, "u"))
        k = min(n, 2 + i % 3)
        m = W.haar_unitary(1 << k, rng) + 0.2 * rng.standard_normal((1 << k, 1 << k))
        ops.append(W.Op(pick(k), m, False, "m"))
        k = min(n, (1, 2, 3, 5, 6)[i % 5])
        d = rng.standard_normal(1 << k) + 1j * rng.standard_normal(1 << k)
        d[0] = 0.0
        d[-1] *= 1e-3
        ops.append(W.Op(pick(k), np.diag(d), True, "d"))
    return ops


@pytest.mark.parametrize("n", [3, 8, 12, 13, 16])
@pytest.mark.parametrize("kmax", [1, 3])
def test_operators_that_are_not_unitary(q, n, kmax):
    """Against the oracle in up to four stretches, each from a state of norm one,
    relative to the norm reached (a stretch whose projectors leave nothing: to one)."""
    rng = np.random.default_rng(10 * n + kmax)
    opts = q.make_opts(planner=q.QSA_PLAN_DP, kmax=kmax, kmax_diag=min(n, 8), kmax_prod=3 if kmax == 1 and n > 3 else 0)
    psi = W.random_state(n, seed=n).astype(np.complex64)
    for _ in range(4):
        ops = _general_ops(n, rng)[:25]
        want = psi.astype(np.complex128)
        for o in ops:
            oracle.apply(want, o.targets, o.matrix)
        st = GState(q, torch, n, init=psi)
        try:
            stats = q.qsa_apply_circuit(st.h, ops, opts)
            assert stats["passes"] < stats["blocks"] or stats["blocks"] == 1   # one dense block on three qubits
            got = st.logical()
        finally:
            st.close()
        norm = np.linalg.norm(want)
        assert np.linalg.norm(got - want) <= 1e-5 * (norm if norm > 0 else 1.0)
        if norm == 0:
            break
        psi = (want / norm).astype(np.complex64)
