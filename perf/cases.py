"""The work that programs built on this library have it do, as measurable cases.

A case is one pass through the public entry points: a compiled circuit, a few
operators called one by one, a change of layout, a read-out, a batch of noisy
trajectories, a density-matrix step or a training step of the cost model.  The
sizes are those of the library's own workloads (the 12-qubit brick circuit, the
QFT + random-layer circuit, the 30-qubit QAOA circuit, width-5/6 operators,
20-qubit trajectories, noisy density matrices, the planner's network) and odd
sizes around them.  ``exact`` recomputes a case in FP64 with plain torch.

Samples drawn from a state that the same pass evolved are not returned: a last
bit of one amplitude moves which outcome a draw falls on, so they say nothing
about the pass beyond the state itself, which is returned whole.  Sampling is a
case of its own, on a given state, and returns every outcome and count.
Probabilities and sums of a state that the same pass evolved in FP32 are
returned in FP32: they are no more accurate than that state.
"""
import math

import numpy as np
import torch

import paper_2608_16940_gb300 as q

H = np.array([[1, 1], [1, -1]], dtype=np.complex128) / math.sqrt(2.0)
CZ = np.diag([1, 1, 1, -1]).astype(np.complex128)
SWAP = np.array([[1, 0, 0, 0], [0, 0, 1, 0], [0, 1, 0, 0], [0, 0, 0, 1]], dtype=np.complex128)
PAULIS = [np.eye(2, dtype=np.complex128), np.array([[0, 1], [1, 0]], dtype=np.complex128),
          np.array([[0, -1j], [1j, 0]]), np.diag([1, -1]).astype(np.complex128)]


def listed():
    return [
        # the smallest call: a 12-qubit brick circuit from |0..0>, state and probabilities read back (launch latency)
        {"name": "brick n12", "kind": "brick", "n": 12, "layers": 20},
        # QFT and random one- and two-qubit layers fused to k <= 4 in FP32 on a state that just outgrows the L2
        {"name": "fusion n25", "kind": "fusion", "n": 25, "layers": 3},
        # the whole QAOA step of a variational loop: evolve from |0..0>, norm and one edge's <ZZ>
        {"name": "qaoa n30 p8", "kind": "qaoa", "n": 30, "p": 8},
        # wide fused operators on the tensor cores, mixed low and high targets, the largest state in daily use
        {"name": "wide n30 tf32x3", "kind": "wide", "n": 30, "ops": 4, "tf32x3": True},
        # the same operators for users who ask for strict FP32
        {"name": "wide n26 fp32", "kind": "wide", "n": 26, "ops": 4, "tf32x3": False},
        # a program that applies operators one by one: dense k = 1..4, a diagonal, a product and a layer
        {"name": "gates n27", "kind": "gates", "n": 27, "kdiag": 8, "kprod": 7, "klayer": 9},
        # moving a state to another qubit order and back, and a few explicit bit swaps
        {"name": "layout n28", "kind": "layout", "n": 28, "pairs": 5},
        # every probability in logical order, left on the device, from a state with a permuted layout
        {"name": "probabilities n27", "kind": "probabilities", "n": 27},
        # two expectations and a large number of samples from one state
        {"name": "measure n26 200k", "kind": "measure", "n": 26, "shots": 200000, "masks": 2},
        # noisy trajectories of uneven depth in one launch
        {"name": "batch n20", "kind": "batch", "n": 20, "traj": 128, "dmin": 10, "dmax": 40, "shots": 10000},
        # channels on one, two and three qubits of a density matrix, then its diagonal
        {"name": "density n13", "kind": "density", "n": 13},
        # one minibatch of the planner's cost model: loss, gradients, Adam
        {"name": "train b64", "kind": "train", "batch": 64},
    ]


def draw(rng):
    kind = rng.choice(["brick", "fusion", "qaoa", "wide", "wide", "gates", "gates", "layout", "probabilities",
                       "measure", "measure", "batch", "density", "train"])
    if kind == "brick":
        return {"kind": kind, "n": rng.randint(7, 16), "layers": rng.randint(4, 20)}
    if kind == "fusion":
        return {"kind": kind, "n": rng.randint(13, 25), "layers": rng.randint(1, 3)}
    if kind == "qaoa":
        return {"kind": kind, "n": 2 * rng.randint(6, 14), "p": rng.randint(1, 8)}
    if kind == "wide":
        tf32x3 = rng.random() < 0.5
        return {"kind": kind, "n": rng.randint(14, 29 if tf32x3 else 26), "ops": rng.randint(2, 4), "tf32x3": tf32x3}
    if kind == "gates":
        return {"kind": kind, "n": rng.randint(13, 27), "kdiag": rng.randint(1, 10), "kprod": rng.randint(1, 11),
                "klayer": rng.randint(1, 9)}
    if kind == "layout":
        return {"kind": kind, "n": rng.randint(13, 28), "pairs": rng.randint(1, 6)}
    if kind == "probabilities":
        return {"kind": kind, "n": rng.randint(12, 27)}
    if kind == "measure":
        return {"kind": kind, "n": rng.randint(12, 26), "shots": int(round(10 ** rng.uniform(2.0, 5.3))),
                "masks": rng.randint(0, 4)}
    if kind == "batch":
        n = rng.randint(10, 20)
        traj = min(256, (1 << 27) >> n)
        return {"kind": kind, "n": n, "traj": rng.randint(max(1, traj // 4), traj), "dmin": rng.randint(2, 10),
                "dmax": rng.randint(12, 40), "shots": int(round(10 ** rng.uniform(2.0, 4.0)))}
    if kind == "density":
        return {"kind": kind, "n": rng.randint(6, 13)}
    return {"kind": kind, "batch": int(round(10 ** rng.uniform(1.2, 3.6)))}


# ---- inputs ---------------------------------------------------------------------


class Op:
    """One circuit operation in the shape the binding takes."""

    def __init__(self, targets, matrix, diag=False):
        self.targets, self.matrix, self.diag = tuple(int(t) for t in targets), matrix, diag


def _haar(count, d, rng):
    """``count`` Haar-random d x d unitaries."""
    z = rng.standard_normal((count, d, d)) + 1j * rng.standard_normal((count, d, d))
    u, r = np.linalg.qr(z)
    ph = np.diagonal(r, axis1=1, axis2=2)
    return u * (ph / np.abs(ph))[:, None, :]


def _zz(g):
    return np.diag(np.exp(-0.5j * g * np.array([1, -1, -1, 1])))


def _rx(b):
    c, s = math.cos(b / 2), math.sin(b / 2)
    return np.array([[c, -1j * s], [-1j * s, c]], dtype=np.complex128)


def _matching(n, rng):
    p = rng.permutation(n)
    return [(int(p[2 * i]), int(p[2 * i + 1])) for i in range(n // 2)]


def _three_regular(n, rng):
    while True:
        pairs = rng.permutation(np.repeat(np.arange(n), 3)).reshape(-1, 2)
        edges = {(int(min(a, b)), int(max(a, b))) for a, b in pairs if a != b}
        if len(edges) == 3 * n // 2:
            return sorted(edges)


def _brick_ops(n, layers, rng):
    us = _haar(n * layers, 2, rng)
    ops = []
    for l in range(layers):
        ops += [Op((j,), us[l * n + j]) for j in range(n)]
        ops += [Op((j, j + 1), CZ, True) for j in range(l % 2, n - 1, 2)]
    return ops


def _fusion_ops(n, layers, rng):
    ops = []
    for j in range(n - 1, -1, -1):
        ops.append(Op((j,), H))
        ops += [Op((i, j), np.diag([1, 1, 1, np.exp(1j * math.pi / (1 << (j - i)))]), True) for i in range(j - 1, -1, -1)]
    ops += [Op((i, n - 1 - i), SWAP) for i in range(n // 2)]
    for _ in range(layers):
        u2, u4 = _haar(n, 2, rng), _haar(n // 2, 4, rng)
        ops += [Op((j,), u2[j]) for j in range(n)]
        ops += [Op(ab, u4[i]) for i, ab in enumerate(_matching(n, rng))]
    return ops


def _qaoa_ops(n, p, rng):
    edges = _three_regular(n, rng)
    gam, bet = rng.uniform(0, 2 * math.pi, p), rng.uniform(0, 2 * math.pi, p)
    ops = [Op((j,), H) for j in range(n)]
    for l in range(p):
        ops += [Op(e, _zz(gam[l]), True) for e in edges]
        ops += [Op((j,), _rx(bet[l])) for j in range(n)]
    return ops, edges


def _interleaved(n):
    sizes = [len(range(g, n, 3)) for g in range(3)]
    return [sum(sizes[:j % 3]) + j // 3 for j in range(n)]


def _wide_ops(n, count, rng):
    return [Op(rng.permutation(n)[:5 + i % 2], _haar(1, 32 << (i % 2), rng)[0]) for i in range(count)]


def _gates(case, rng):
    """Operators in the order they are called: ("fused", op), ("diag", targets,
    entries), ("product", targets, factors), ("layer", diagonal ops, targets,
    factors).  The factors of a layer sit on qubits that fit one tile."""
    n = case["n"]
    calls = [("fused", Op(rng.permutation(n)[:k], _haar(1, 1 << k, rng)[0])) for k in (1, 2, 3, 4)]
    k = case["kdiag"]
    calls.append(("diag", rng.permutation(n)[:k], np.exp(1j * rng.uniform(0, 2 * math.pi, 1 << k))))
    k = case["kprod"]
    calls.append(("product", rng.permutation(n)[:k], _haar(k, 2, rng)))
    k = case["klayer"]
    dops = [Op(ab, _zz(rng.uniform(0, 2 * math.pi)), True) for ab in _matching(n, rng)]
    calls.append(("layer", dops, rng.permutation(n)[:k], np.stack([_rx(b) for b in rng.uniform(0, 2 * math.pi, k)])))
    return calls


def _trajectory(n, depth, rng, p=1e-3):
    """Layers of one noisy trajectory: (one-qubit unitaries with their Pauli
    branches multiplied in, first qubit of the CZ brick, two-qubit Pauli
    branches after it), and the same as a list of ops."""
    layers, ops = [], []
    for l in range(depth):
        us, q0 = _haar(n, 2, rng), l % 2
        hit = rng.random(n) < p
        ops += [Op((j,), us[j].copy()) for j in range(n)]
        for j in np.nonzero(hit)[0]:
            P = PAULIS[1 + int(rng.integers(0, 3))]
            ops.append(Op((int(j),), P))
            us[j] = P @ us[j]
        pauli = []
        for j in range(q0, n - 1, 2):
            ops.append(Op((j, j + 1), CZ, True))
            if rng.random() < p:
                s = 1 + int(rng.integers(0, 15))
                pauli.append(Op((j, j + 1), np.kron(PAULIS[s >> 2], PAULIS[s & 3])))
        ops += pauli
        layers.append((us, q0, pauli))
    return layers, ops


def _trajectories(case, rng):
    return [_trajectory(case["n"], int(d), rng)
            for d in rng.integers(case["dmin"], case["dmax"] + 1, size=case["traj"])]


def _channels(n, rng):
    """(targets, Kraus operators, precision): amplitude damping, two-qubit
    depolarising noise after a random gate, a random three-qubit channel."""
    g = 0.1
    damp = np.array([[[1, 0], [0, math.sqrt(1 - g)]], [[0, math.sqrt(g)], [0, 0]]], dtype=np.complex128)
    u, p = _haar(1, 4, rng)[0], 0.01
    depol = np.stack([(math.sqrt(1 - 15 * p / 16) if s == 0 else math.sqrt(p / 16)) *
                      np.kron(PAULIS[s >> 2], PAULIS[s & 3]) @ u for s in range(16)])
    iso = _haar(1, 24, rng)[0][:, :8].reshape(3, 8, 8)   # an isometry cut into three Kraus operators
    return [(rng.permutation(n)[:1], damp, q.QSA_PREC_FP32), (rng.permutation(n)[:2], depol, q.QSA_PREC_FP32),
            (rng.permutation(n)[:3], iso, q.QSA_PREC_TF32X3)]


def _random_state(n, seed, dtype=torch.complex64):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    x = torch.randn(2 << n, device="cuda", generator=g)
    x /= torch.linalg.vector_norm(x, dtype=torch.float64).item()
    return torch.view_as_complex(x.view(-1, 2)).to(dtype)


def _random_density(n, seed):
    """vec(rho), column-major, of a mixture of four random pure states."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    a = torch.randn(1 << n, 4, 2, device="cuda", dtype=torch.float64, generator=g)
    a = torch.view_as_complex(a)
    a /= torch.linalg.vector_norm(a)
    return (a @ a.mH).T.contiguous().view(-1).to(torch.complex64)


def _training(batch, seed):
    """Parameters in mid-training, features of random passes and their log times."""
    rng = np.random.default_rng(seed)
    X = np.zeros((batch, q.MLP_IN), dtype=np.float32)
    for row in X:
        n, k = int(rng.integers(20, 31)), int(rng.integers(1, 7))
        row[0] = k / 6
        row[1 + rng.permutation(n)[:k]] = 1
        row[35] = n / 34
    t = rng.standard_normal(batch).astype(np.float32)
    p = q.qsa_costmodel_init(int(seed)) + rng.normal(0, 0.01, q.MLP_PARAMS).astype(np.float32)
    m = rng.normal(0, 1e-2, q.MLP_PARAMS).astype(np.float32)
    v = rng.uniform(1e-4, 1e-2, q.MLP_PARAMS).astype(np.float32)
    return {"p": p, "X": X, "t": t, "m": m, "v": v}


class State:
    """A library state over a torch-owned buffer, the plan kept with it."""

    def __init__(self, n, buf, init_zero=0):
        self.n, self.buf, self.plan = n, buf, None
        self.h = q.qsa_state_create_ex(n, buf.data_ptr(), buf.numel() * 8, torch.cuda.current_stream().cuda_stream,
                                       init_zero)

    def __del__(self):
        if self.plan:
            q.qsa_plan_destroy(self.plan)
        q.qsa_state_destroy(self.h)


class Batch:
    def __init__(self, n, trajs):
        self.h = q.qsa_batch_create(n, trajs, q.make_opts(planner=q.QSA_PLAN_DP, kmax=4))

    def __del__(self):
        q.qsa_batch_destroy(self.h)


def prepare(case, seed):
    kind, rng = case["kind"], np.random.default_rng(seed)
    if kind in ("brick", "qaoa"):
        n = case["n"]
        st = State(n, torch.empty(1 << n, dtype=torch.complex64, device="cuda"), 1)
        if kind == "brick":
            st.plan = q.qsa_plan_create(_brick_ops(n, case["layers"], rng), n, q.qsa_plan_opts_default())
            return {"case": case, "st": st, "probs": torch.empty(1 << n, dtype=torch.float64, device="cuda")}
        ops, edges = _qaoa_ops(n, case["p"], rng)
        opts = q.make_opts(planner=q.QSA_PLAN_DP, kmax=6, kmax_diag=12, layer=1, zero_init=1,
                           precision=q.QSA_PREC_TF32X3)
        st.plan = q.qsa_plan_create(ops, n, opts, layout=_interleaved(n))
        return {"case": case, "st": st, "masks": [0, (1 << edges[0][0]) | (1 << edges[0][1])]}
    if kind in ("fusion", "wide"):
        n = case["n"]
        st = State(n, _random_state(n, seed))
        if kind == "fusion":
            ops, opts = _fusion_ops(n, case["layers"], rng), q.make_opts(planner=q.QSA_PLAN_DP, kmax=4)
        else:
            ops = _wide_ops(n, case["ops"], rng)
            opts = q.make_opts(planner=q.QSA_PLAN_PER_GATE, kmax=6, kmax_diag=6,
                               precision=q.QSA_PREC_TF32X3 if case["tf32x3"] else q.QSA_PREC_FP32)
        st.plan = q.qsa_plan_create(ops, n, opts)
        return {"case": case, "st": st}
    if kind == "gates":
        return {"case": case, "st": State(case["n"], _random_state(case["n"], seed)), "calls": _gates(case, rng)}
    if kind == "layout":
        n = case["n"]
        a, b = (rng.permutation(n).tolist() for _ in range(2))
        p = rng.permutation(n)[:2 * case["pairs"]].tolist()
        return {"case": case, "st": State(n, _random_state(n, seed)), "layouts": (a, b),
                "pairs": (p[::2], p[1::2])}
    if kind in ("probabilities", "measure"):
        n = case["n"]
        st = State(n, torch.zeros(1 << n, dtype=torch.complex64, device="cuda"), 1)
        q.qsa_set_layout(st.h, rng.permutation(n).tolist(), materialise=0)
        st.buf.copy_(_random_state(n, seed))
        if kind == "probabilities":
            return {"case": case, "st": st, "probs": torch.empty(1 << n, dtype=torch.float64, device="cuda")}
        # the histogram goes into arrays of the program's own, one slot per shot, zero beyond the distinct outcomes
        return {"case": case, "st": st, "masks": _masks(n, case["masks"], rng), "seed": int(seed),
                "outcomes": np.zeros(case["shots"], dtype=np.int64), "counts": np.zeros(case["shots"], dtype=np.int64)}
    if kind == "batch":
        b = Batch(case["n"], [ops for _, ops in _trajectories(case, rng)])
        return {"case": case, "batch": b, "seed": int(seed),
                "states": torch.empty(case["traj"], 1 << case["n"], dtype=torch.complex64, device="cuda")}
    if kind == "density":
        return {"case": case, "st": State(2 * case["n"], _random_density(case["n"], seed)),
                "channels": _channels(case["n"], rng)}
    d = {k: torch.from_numpy(v).cuda() for k, v in _training(case["batch"], seed).items()}
    d["g"], d["loss"] = torch.empty_like(d["p"]), torch.empty(1, device="cuda")
    d["ws"] = torch.empty(q.qsa_mlp_workspace_bytes(case["batch"]) // 4, device="cuda")
    d["case"] = case
    return d


def _masks(n, count, rng):
    return [0, 3, 1 << (n - 1), int(rng.integers(1, 1 << n))][:count]


# ---- one pass -------------------------------------------------------------------


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        s = torch.cuda.current_stream().cuda_stream
        p, X, t, g = (state[k].data_ptr() for k in ("p", "X", "t", "g"))
        q.qsa_mlp_loss_grad(p, X, t, case["batch"], g, state["loss"].data_ptr(), state["ws"].data_ptr(), s)
        q.qsa_mlp_adam_step(p, g, state["m"].data_ptr(), state["v"].data_ptr(), q.MLP_PARAMS, 100, stream=s)
        return {k: state[k] for k in ("loss", "g", "p", "m", "v")}
    if kind == "batch":
        x = state["states"]
        q.qsa_batch_run(state["batch"].h, x.data_ptr(), x.numel() * 8, case["shots"], state["seed"], 0, 1,
                        torch.cuda.current_stream().cuda_stream)
        return x
    st = state["st"]
    h = st.h
    if kind == "brick":
        q.qsa_plan_execute_from_zero(h, st.plan)
        norm = q.qsa_probabilities_device(h, state["probs"].data_ptr())
        return {"state": st.buf, "probs": state["probs"].float(), "norm": np.float32(norm)}
    if kind == "qaoa":
        q.qsa_plan_execute_from_zero(h, st.plan)
        return {"z": np.float32(q.qsa_expectation_z_batch(h, state["masks"])), "state": st.buf}
    if kind in ("fusion", "wide"):
        q.qsa_plan_execute(h, st.plan)
        return st.buf
    if kind == "gates":
        for call in state["calls"]:
            if call[0] == "fused":
                q.qsa_apply_fused(h, call[1].targets, call[1].matrix)
            elif call[0] == "diag":
                q.qsa_apply_diag(h, call[1], call[2])
            elif call[0] == "product":
                q.qsa_apply_product(h, call[1], call[2])
            else:
                q.qsa_apply_layer(h, call[1], call[2], call[3])
        return st.buf
    if kind == "layout":
        for lay in state["layouts"]:
            q.qsa_set_layout(h, lay)
        q.qsa_permute_bits(h, *state["pairs"])
        return {"state": st.buf, "layout": np.array(q.qsa_get_layout(h))}
    if kind == "probabilities":
        norm = q.qsa_probabilities_device(h, state["probs"].data_ptr())
        return {"probs": state["probs"], "norm": norm}
    if kind == "measure":
        z, vals, cnts = q.qsa_measure(h, state["masks"], case["shots"], state["seed"])
        for name, got in (("outcomes", vals), ("counts", cnts)):
            state[name][:len(got)] = got
            state[name][len(got):] = 0
        return {"z": z, "outcomes": state["outcomes"], "counts": state["counts"]}
    n = case["n"]
    for targets, kraus, prec in state["channels"]:
        q.qsa_dm_apply_channel(h, n, targets, kraus, prec)
    probs, trace = q.qsa_dm_probabilities(h, n)
    return {"rho": st.buf, "probs": probs.astype(np.float32), "trace": np.float32(trace)}


def work(case):
    """Bytes: the state read once (where it is an input) and written once, the
    read-out written once.  Flops: the operators as given, 8 per complex
    multiply-add (a dense k-qubit one: 8 * 2^k per amplitude; a diagonal: 6)."""
    kind = case["kind"]
    if kind == "train":
        return {"bytes": 4 * (q.MLP_PARAMS * 7 + case["batch"] * (q.MLP_IN + 1)), "flops": 6 * q.MLP_PARAMS * case["batch"]}
    n = case["n"]
    amps = 1 << n
    if kind == "brick":
        return {"bytes": 16 * amps, "flops": case["layers"] * amps * (16 * n + 3 * n)}
    if kind == "fusion":
        return {"bytes": 16 * amps,
                "flops": amps * (16 * n + 3 * n * (n - 1) + case["layers"] * (16 * n + 32 * (n // 2)))}
    if kind == "qaoa":
        return {"bytes": 8 * amps, "flops": amps * (16 * n * (case["p"] + 1) + 9 * n * case["p"])}
    if kind == "wide":
        return {"bytes": 16 * amps, "flops": amps * sum(256 << (i % 2) for i in range(case["ops"]))}
    if kind == "gates":
        return {"bytes": 16 * amps, "flops": amps * (8 * 30 + 6 + 16 * case["kprod"] + 3 * n + 16 * case["klayer"])}
    if kind == "layout":
        return {"bytes": 16 * amps, "flops": 0}
    if kind == "probabilities":
        return {"bytes": 16 * amps, "flops": 3 * amps}
    if kind == "measure":
        return {"bytes": 8 * amps + 16 * case["shots"], "flops": amps * (4 + 2 * case["masks"])}
    if kind == "batch":
        depth = (case["dmin"] + case["dmax"]) / 2
        return {"bytes": 8 * amps * case["traj"], "flops": case["traj"] * depth * amps * (16 * n + 3 * n)}
    amps = 1 << (2 * n)
    return {"bytes": 16 * amps, "flops": amps * 8 * (4 + 16 + 64)}


# ---- the same in FP64 -----------------------------------------------------------


def _apply64(psi, n, pos, M):
    """M on bit positions pos (bit j of M's index = position pos[j])."""
    k = len(pos)
    M = torch.as_tensor(np.ascontiguousarray(M, dtype=np.complex128), device=psi.device)
    shape, axis, prev = [], {}, n
    for j in sorted(range(k), key=lambda j: -pos[j]):
        axis[j] = len(shape) + 1
        shape += [1 << (prev - pos[j] - 1), 2]
        prev = pos[j]
    shape.append(1 << prev)
    x = psi.view(shape)
    if np.count_nonzero(M.cpu().numpy() - np.diag(np.diagonal(M.cpu().numpy()))) == 0 and k <= 2:
        return _diag64(psi, n, pos, torch.diagonal(M))
    front = [axis[j] for j in range(k - 1, -1, -1)]
    perm = front + [i for i in range(len(shape)) if i not in front]
    y = M @ x.permute(perm).reshape(1 << k, -1)
    return y.view([shape[i] for i in perm]).permute(np.argsort(perm).tolist()).reshape(-1)


def _diag64(psi, n, pos, d):
    """Multiplies in place by the diagonal d over bit positions pos."""
    k = len(pos)
    shape, bshape, prev = [], [], n
    order = sorted(range(k), key=lambda j: -pos[j])
    for j in order:
        shape += [1 << (prev - pos[j] - 1), 2]
        bshape += [1, 2]
        prev = pos[j]
    d = torch.as_tensor(d, dtype=torch.complex128, device=psi.device).view([2] * k)
    d = d.permute([k - 1 - j for j in order]).reshape(bshape + [1])
    psi.view(shape + [1 << prev]).mul_(d)
    return psi


def _ops64(psi, n, ops, L=None):
    for o in ops:
        psi = _apply64(psi, n, [L[t] if L is not None else t for t in o.targets], o.matrix)
    return psi


def _zero64(n):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1
    return psi


def _prob64(psi):
    x = torch.view_as_real(psi.to(torch.complex128))
    return x[:, 0] ** 2 + x[:, 1] ** 2


def _z64(p, n, phys_mask):
    """sum of (-1)^popcount(y & phys_mask) p_y."""
    for b in range(n):
        p = p.view(-1, 2)
        p = p[:, 0] - p[:, 1] if (phys_mask >> b) & 1 else p.sum(1)
    return float(p)


def _logical64(x, n, L):
    """x in stored order -> logical order (bit L[j] of the stored index is bit j)."""
    return _bits64(x, [L[j] for j in range(n)])


def _bits64(x, src):
    """out[i] = x[y] with bit src[j] of y = bit j of i."""
    n = len(src)
    i = torch.arange(1 << n, device=x.device)
    y = torch.zeros_like(i)
    for j in range(n):
        y |= ((i >> j) & 1) << src[j]
    return x[y]


def exact(case, seed):
    kind, rng = case["kind"], np.random.default_rng(seed)
    if kind == "train":
        d = {k: torch.from_numpy(v).cuda().double() for k, v in _training(case["batch"], seed).items()}
        p = d["p"].requires_grad_()
        w1, b1, w2, b2, w3, b3 = torch.split(p, [64 * 37, 64, 64 * 64, 64, 64, 1])
        a = torch.relu(d["X"] @ w1.view(64, 37).T + b1)
        a = torch.relu(a @ w2.view(64, 64).T + b2)
        loss = ((a @ w3 + b3 - d["t"]) ** 2).mean()
        loss.backward()
        g = p.grad
        m, v = 0.9 * d["m"] + 0.1 * g, 0.999 * d["v"] + 0.001 * g * g
        out = p.detach() - 1e-3 * (m / (1 - 0.9 ** 100)) / (torch.sqrt(v / (1 - 0.999 ** 100)) + 1e-8)
        return {"loss": loss.detach().view(1), "g": g, "p": out, "m": m, "v": v}
    n = case["n"]
    if kind == "brick":
        psi = _ops64(_zero64(n), n, _brick_ops(n, case["layers"], rng))
        p = _prob64(psi)
        return {"state": psi, "probs": p, "norm": float(p.sum())}
    if kind == "fusion":
        return _ops64(_random_state(n, seed, torch.complex128), n, _fusion_ops(n, case["layers"], rng))
    if kind == "wide":
        return _ops64(_random_state(n, seed, torch.complex128), n, _wide_ops(n, case["ops"], rng))
    if kind == "qaoa":
        ops, edges = _qaoa_ops(n, case["p"], rng)
        L = _interleaved(n)
        psi = torch.full((1 << n,), 2.0 ** (-n / 2), dtype=torch.complex128, device="cuda")
        ne = len(edges)
        cut = torch.zeros(1 << n, dtype=torch.int8, device="cuda")   # edges whose ends differ
        for a, b in edges:
            hi, lo = max(L[a], L[b]), min(L[a], L[b])
            x = cut.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
            x[:, 0, :, 1] += 1
            x[:, 1, :, 0] += 1
        for l in range(case["p"]):
            o = n + l * (ne + n)
            same, diff = np.diagonal(ops[o].matrix)[:2]
            tab = torch.tensor([same ** (ne - c) * diff ** c for c in range(ne + 1)], device="cuda")
            for lo in range(0, 1 << n, 1 << 26):
                psi[lo:lo + (1 << 26)] *= tab[cut[lo:lo + (1 << 26)].long()]
            c, s = ops[o + ne].matrix[0]
            for pos in range(n):
                x = psi.view(-1, 2, 1 << pos)
                x0 = x[:, 0].clone()
                x[:, 0].mul_(c.real).add_(x[:, 1], alpha=complex(s))
                x[:, 1].mul_(c.real).add_(x0, alpha=complex(s))
                del x0
        p = _prob64(psi)
        masks = [0, (1 << L[edges[0][0]]) | (1 << L[edges[0][1]])]
        return {"z": np.array([_z64(p, n, m) for m in masks]), "state": psi}
    if kind == "gates":
        psi = _random_state(n, seed, torch.complex128)
        for call in _gates(case, rng):
            if call[0] == "fused":
                psi = _ops64(psi, n, [call[1]])
            elif call[0] == "diag":
                psi = _diag64(psi, n, call[1].tolist(), call[2])
            else:
                if call[0] == "layer":
                    psi = _ops64(psi, n, call[1])
                psi = _ops64(psi, n, [Op((t,), f) for t, f in zip(call[-2], call[-1])])
        return psi
    if kind == "layout":
        b = [rng.permutation(n).tolist() for _ in range(2)][1]
        p = rng.permutation(n)[:2 * case["pairs"]].tolist()
        swap = dict(list(zip(p[::2], p[1::2])) + list(zip(p[1::2], p[::2])))
        L = [swap.get(x, x) for x in b]
        inv = np.argsort(L).tolist()   # position y holds logical qubit inv[y]
        return {"state": _bits64(_random_state(n, seed, torch.complex128), inv), "layout": None}
    if kind in ("probabilities", "measure"):
        L = rng.permutation(n).tolist()
        p = _prob64(_random_state(n, seed, torch.complex128))
        if kind == "probabilities":
            return {"probs": _logical64(p, n, L), "norm": float(p.sum())}
        masks = _masks(n, case["masks"], rng)
        phys = [sum(1 << L[j] for j in range(n) if (m >> j) & 1) for m in masks]
        return {"z": [_z64(p, n, m) for m in phys], "outcomes": None, "counts": None}
    if kind == "batch":
        return _batch64(case, rng)
    rho = _random_density(n, seed).to(torch.complex128)
    for targets, kraus, _ in _channels(n, rng):
        S = sum(np.kron(e.conj(), e) for e in kraus.reshape(-1, 1 << len(targets), 1 << len(targets)))
        rho = _apply64(rho, 2 * n, [int(t) for t in targets] + [int(t) + n for t in targets], S)
    diag = rho.view(1 << n, 1 << n).diagonal().real.clone()
    return {"rho": rho, "probs": diag, "trace": float(diag.sum())}


def _batch64(case, rng):
    """Each trajectory layer by layer: the one-qubit unitaries as Kronecker
    products over groups of five qubits, the CZ brick as a sign."""
    n = case["n"]
    idx = torch.arange(1 << n, device="cuda")
    sign = []
    for q0 in (0, 1):
        par = torch.zeros_like(idx)
        for j in range(q0, n - 1, 2):
            par ^= (idx >> j) & (idx >> (j + 1)) & 1
        sign.append((1 - 2 * par).to(torch.float64))
    out = torch.empty(case["traj"], 1 << n, dtype=torch.complex128, device="cuda")
    for i, (layers, _) in enumerate(_trajectories(case, rng)):
        psi = _zero64(n)
        for us, q0, pauli in layers:
            for j in range(0, n, 5):
                M = np.ones((1, 1))
                for u in us[j:j + 5]:
                    M = np.kron(u, M)
                M = torch.from_numpy(M).cuda()
                d = M.shape[0]
                psi = torch.matmul(M, psi.view(-1, d, 1 << j)).reshape(-1)
            psi = psi * sign[q0]
            for o in pauli:
                psi = _apply64(psi, n, list(o.targets), o.matrix)
        out[i] = psi
    return out
