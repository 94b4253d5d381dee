"""Group passes at the edges of what they accept: groups that multiply to the
identity and so have no pass.  Same tolerance as the other group tests (1e-5 on
fidelity and amplitudes, FP32 sums of at most 32 terms over a few blocks)."""
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
