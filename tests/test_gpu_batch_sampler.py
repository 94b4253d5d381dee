"""Batched trajectories whose shots are drawn and sorted together, bit for bit
against the oracle's sampler on the states that the run left (Philox stream =
trajectory), around the number of shots where that begins: one and several
blocks of 1024 amplitudes per state, a number of trajectories that is no power
of two, one trajectory, an empty one, and direct launches next to the graph."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_16940_gb300 as q
    return q


@pytest.mark.parametrize("n,n_traj,shots", [(9, 20, 2000), (10, 9, 2000), (10, 16, 1023), (10, 16, 1024), (11, 3, 16384),
                                            (13, 1, 16384), (14, 37, 1000), (18, 5, 10000)])
def test_batch_counts_match_oracle(q, n, n_traj, shots):
    trajs = [[] if t == 1 else W.trajectory_circuit(n, 3, np.random.default_rng([n, t]), 0.05)[0] for t in range(n_traj)]
    b = q.qsa_batch_create(n, trajs, q.make_opts(planner=q.QSA_PLAN_DP, kmax=4))
    states = torch.zeros(n_traj << n, dtype=torch.complex64, device="cuda:0")
    try:
        for use_graph in (0, 1):
            q.qsa_batch_run(b, states.data_ptr(), states.numel() * 8, shots, 77, 0, use_graph)
            res = q.qsa_batch_counts(b, n_traj, shots)
            psi = states.view(n_traj, -1).cpu().numpy()
            for t in range(n_traj):
                want, cnt = oracle.sample_counts(psi[t].astype(np.complex128), list(range(n)), shots, 77, t)
                assert np.array_equal(res[t][0], want) and np.array_equal(res[t][1], cnt), (use_graph, t)
    finally:
        q.qsa_batch_destroy(b)
