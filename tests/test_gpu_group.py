"""Group passes (several fused blocks in one pass over the state) against the
oracle: states below, at and above one tile of 2^12 amplitudes, dense blocks of
every width on low and high positions, diagonal blocks whose qubits lie in and
outside the tile, product factors, permuted layouts, and plans run from
|0...0> on a buffer that holds something else.  FP32 sums of at most 16 terms
per block and a few dozen blocks stay far below the suite's 1e-5."""
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


def _mixed_ops(n, count, rng):
    """Dense k = 1..4 and flagged diagonal k = 1..6 operators on random targets."""
    ops = []
    for _ in range(count):
        diag = rng.random() < 0.4
        k = int(rng.integers(1, min(n, 6 if diag else 4) + 1))
        t = tuple(int(v) for v in rng.choice(n, size=k, replace=False))
        if diag:
            ops.append(W.Op(t, np.diag(np.exp(1j * rng.uniform(0, 2 * np.pi, 1 << k))), True, "d"))
        else:
            ops.append(W.Op(t, W.haar_unitary(1 << k, rng), False, "u"))
    return ops


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 11, 12, 13, 14, 17, 20])
@pytest.mark.parametrize("planner", ["greedy", "dp"])
def test_grouped_plan_matches_oracle(q, n, planner):
    rng = np.random.default_rng(100 + n)
    ops = _mixed_ops(n, 60, rng)
    L = [int(v) for v in rng.permutation(n)]
    opts = q.make_opts(planner={"greedy": q.QSA_PLAN_GREEDY, "dp": q.QSA_PLAN_DP}[planner], kmax=4, kmax_diag=6,
                       kmax_prod=4 if n > 4 else 0)
    plan = q.qsa_plan_create(ops, n, opts, layout=L)
    psi = W.random_state(n, seed=n).astype(np.complex64)
    st = GState(q, torch, n, init=psi)
    try:
        # arbitrary contents, identity layout: the plan's blocks one by one (its passes are for another layout)
        stats = q.qsa_plan_execute(st.h, plan)
        want = psi.astype(np.complex128)
        for o in ops:
            oracle.apply(want, o.targets, o.matrix)
        check_close(want, st.logical())
        # from |0...0> in the plan's layout: group passes, the first one generating the state
        blocks = stats["blocks"]
        stats = q.qsa_plan_execute_from_zero(st.h, plan)
        assert q.qsa_get_layout(st.h) == L and stats["blocks"] == blocks
        if blocks > 3:
            assert stats["passes"] < blocks
        check_close(oracle.run_circuit(n, ops), st.logical())
        # and again from what that left
        q.qsa_plan_execute(st.h, plan)
        check_close(oracle.run_circuit(n, ops + ops), st.logical())
    finally:
        st.close()
        q.qsa_plan_destroy(plan)
