"""The work that a user of this package has it do, as cases that can be timed.

Every case is one pass through public entry points (tnq.contract_sliced,
tnq.contract_sliced_noalloc, tnq.amplitudes_batch, learned.train,
learned.gpu_grad) on what a program has in hand at that point: a plan, a
device workspace and the bitstrings, or the training rows. A circuit belongs to
the case (a plan is made once per circuit); bitstrings and rows come from the
seed, and so do the tensors of a general network.

The contraction computes its slices in complex64 (32-bit parts) and adds them
in 64 bits. Its values are returned here as complex64, the type that they are
computed in.
"""
import numpy as np
import torch

from paper_2004_10892_gb300 import inputs, learned, shard, tnq

PRECISIONS = {"c64": tnq.PREC_C64, "bf16x3": tnq.PREC_SPLIT_BF16, "tf32x3": tnq.PREC_SPLIT_TF32}


# ---- the cases -------------------------------------------------------------
def _amplitude(rows, cols, depth, circuit=0, **kw):
    """Slices of one amplitude of a grid circuit: rank `rank`'s share of them among `world` (all, for 0 of 1), or
    the first `chunk` of that share (a worker takes a long share in chunks)."""
    case = dict(kind="amplitude", rows=rows, cols=cols, depth=depth, circuit=circuit, precision="c64", max_bag=28,
                min_p=0, max_p=40, reorder=0, trials=1, rank=0, world=1, chunk=0, per_slice=True,
                noalloc=False)
    return dict(case, **kw)


def _serve(circuits, bitstrings, smallest, largest, depth_from, depth_to, **kw):
    """One batched request: `bitstrings` amplitudes of each of several circuits on mixed square grids."""
    case = dict(kind="serve", circuits=circuits, bitstrings=bitstrings, smallest=smallest, largest=largest,
                depth_from=depth_from, depth_to=depth_to, circuit=0, precision="c64", max_bag=26, max_p=30, reorder=1,
                workspace_gb=4)
    return dict(case, **kw)


def _lattice(rows, cols, dim, **kw):
    """A closed lattice network with indices of `dim` values, every slice."""
    case = dict(kind="lattice", rows=rows, cols=cols, dim=dim, precision="c64", max_bag=20, min_p=0, max_p=10)
    return dict(case, **kw)


def listed():
    return [
        # the smallest amplitude anyone asks for: a 16-qubit check circuit, bound by latency
        dict(_amplitude(4, 4, 16, max_bag=0, max_p=0, per_slice=False), name="amp_4x4_d16"),
        # one amplitude in a loop that may not allocate (the deployment variant)
        dict(_amplitude(5, 5, 20, circuit=3, max_bag=0, max_p=0, per_slice=False, noalloc=True),
             name="noalloc_5x5_d20"),
        # the 6x6 configuration: sixteen slices that all fit one batch
        dict(_amplitude(6, 6, 24, max_bag=24, min_p=4, max_p=8), name="slices_6x6_d24"),
        # the 7x7 benchmark circuit and plan in each precision
        dict(_amplitude(7, 7, 32, precision="bf16x3", reorder=1, trials=32), name="amp_7x7_d32_bf16x3"),
        dict(_amplitude(7, 7, 32, precision="tf32x3", reorder=1, trials=32), name="amp_7x7_d32_tf32x3"),
        dict(_amplitude(7, 7, 32, reorder=1, trials=32), name="amp_7x7_d32_c64"),
        # one worker's share (37 of 256 slices, no power of two) of the plan that default options make
        dict(_amplitude(7, 7, 32, rank=2, world=7), name="share_7x7_d32_37of256"),
        # a request for many small amplitudes: latency and the number of launches
        dict(_serve(12, 5, 4, 6, 16, 24, circuit=2), name="serve_small_c64"),
        # a request as the serving workload has them: four circuits, 6x6 and 7x7, of very different cost
        dict(_serve(4, 16, 5, 7, 16, 32, precision="bf16x3", workspace_gb=24), name="serve_mixed_bf16x3"),
        # a general network: indices of three values, padded to two binary digits each
        dict(_lattice(6, 6, 3, min_p=2), name="lattice_6x6_L3"),
        # training the slicing proposer: one epoch, and the gradient over all the rows of the 500-circuit set
        dict(kind="train", rows=8256, batch=1024, hidden=128, epochs=1, name="proposer_epoch"),
        dict(kind="grad", rows=162805, hidden=128, name="proposer_grad_162805"),
    ]


def draw(rng):
    """One more case of the ranges above."""
    what = rng.choice(["amplitude"] * 6 + ["noalloc", "serve", "lattice", "train", "grad"])
    circuit = rng.randrange(1, 10000)
    if what == "amplitude":
        rows, cols, depth = rng.randint(4, 7), rng.randint(4, 7), rng.randint(16, 32)
        world = rng.choice([1, 1, 2, 3, 5])
        return _amplitude(rows, cols, depth, circuit, precision=rng.choice(["c64", "bf16x3", "tf32x3"]),
                          max_bag=rng.randint(20, 26), min_p=rng.randint(0, 3), reorder=1, rank=rng.randrange(world),
                          world=world, chunk=rng.randint(17, 32))
    if what == "noalloc":
        return _amplitude(rng.randint(3, 5), rng.randint(4, 6), rng.randint(8, 20), circuit, max_bag=16, chunk=32,
                          noalloc=True)
    if what == "serve":
        return _serve(rng.randint(2, 10), rng.randint(1, 8), 4, 6, 12, 20, circuit=circuit,
                      precision=rng.choice(["c64", "bf16x3"]), max_bag=rng.randint(18, 22))
    if what == "lattice":
        return _lattice(rng.randint(4, 6), rng.randint(4, 6), rng.randint(2, 4), max_bag=18,
                        precision=rng.choice(["c64", "bf16x3"]), min_p=rng.randint(1, 3))
    if what == "train":
        return dict(kind="train", rows=int(2 ** rng.uniform(10, 13.5)), batch=rng.choice([256, 512, 1024]),
                    hidden=rng.choice([32, 64, 128]), epochs=1)
    return dict(kind="grad", rows=int(2 ** rng.uniform(5, 17)), hidden=rng.choice([16, 48, 64, 128]))


# ---- what a program has before the call ---------------------------------------
def _circuit(case):
    return inputs.random_grid_circuit(case["rows"], case["cols"], case["depth"], case["circuit"])


def _plan(case, circ):
    return tnq.Plan(circ, max_bag_log2=case["max_bag"], min_p=case["min_p"], max_p=case["max_p"],
                    precision=PRECISIONS[case["precision"]], reorder_every=case["reorder"], order_trials=case["trials"])


def _range(case, plan):
    begin, end = shard.slice_range(plan.info()["n_slices"], case["rank"], case["world"])
    if end == begin:  # more workers than slices
        begin, end = 0, 1
    return begin, min(end, begin + case["chunk"]) if case["chunk"] else end


def _serve_circuits(case):
    rng = inputs.SplitMix64(case["circuit"] ^ 0x5E5E5E5E)
    circuits = []
    for i in range(case["circuits"]):
        side = case["smallest"] + rng.below(case["largest"] - case["smallest"] + 1)
        depth = case["depth_from"] + 4 * rng.below((case["depth_to"] - case["depth_from"]) // 4 + 1)
        circuits.append(inputs.random_grid_circuit(side, side, depth, case["circuit"] + i))
    return circuits


def _serve_bits(case, circuits, seed):
    return [[inputs.random_bitstring(c.n_qubits, seed * 100003 + i * 1000 + j) for j in range(case["bitstrings"])]
            for i, c in enumerate(circuits)]


def _network(case, seed):
    return inputs.random_lattice_network(case["rows"], case["cols"], case["dim"], seed)


def _network_plan(case, net):
    return tnq.Plan.from_network(net.dims, net.tensors, max_bag_log2=case["max_bag"], min_p=case["min_p"],
                                 max_p=case["max_p"], precision=PRECISIONS[case["precision"]])


def _rows(case, seed):
    rng = np.random.default_rng(seed)
    X = rng.random((case["rows"], learned.features()), dtype=np.float32)
    y = (0.25 + 0.25 * rng.standard_normal(case["rows"])).astype(np.float32)
    return X, y


def _power_of_two(n):
    return 1 << (max(n, 1) - 1).bit_length()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "amplitude":
        circ = _circuit(case)
        plan = _plan(case, circ)
        begin, end = _range(case, plan)
        batch = _power_of_two(end - begin)
        while batch > 1 and plan.workspace_bytes(batch) > 24 << 30:
            batch //= 2
        ws = None
        if not case["noalloc"]:
            ws = torch.empty(plan.workspace_bytes(batch), dtype=torch.uint8, device="cuda")
        return dict(kind=kind, case=case, plan=plan, bits=inputs.random_bitstring(circ.n_qubits, seed), begin=begin,
                    end=end, workspace=ws, batch=batch)
    if kind == "serve":
        circuits = _serve_circuits(case)
        plans = [tnq.Plan(c, max_bag_log2=case["max_bag"], max_p=case["max_p"], reorder_every=case["reorder"],
                          precision=PRECISIONS[case["precision"]]) for c in circuits]
        ws = torch.empty(case["workspace_gb"] << 30, dtype=torch.uint8, device="cuda")
        return dict(kind=kind, plans=plans, bits=_serve_bits(case, circuits, seed), workspace=ws,
                    each=case["bitstrings"])
    if kind == "lattice":
        plan = _network_plan(case, _network(case, seed))
        n = plan.info()["n_slices"]
        ws = torch.empty(plan.workspace_bytes(n), dtype=torch.uint8, device="cuda")
        return dict(kind=kind, plan=plan, end=n, workspace=ws)
    X, y = _rows(case, seed)
    if kind == "train":  # host rows: learned.train moves them itself
        return dict(kind=kind, case=case, X=X, y=y, seed=seed)
    params = torch.from_numpy(learned.init_params(seed, case["hidden"])).cuda()
    return dict(kind=kind, case=case, X=torch.from_numpy(X).cuda(), y=torch.from_numpy(y).cuda(), params=params)


def _single(values):
    return np.asarray(values, np.complex128).reshape(-1).astype(np.complex64)


def run(state):
    kind = state["kind"]
    if kind == "amplitude":
        case, span = state["case"], (state["begin"], state["end"])
        if case["noalloc"]:
            out = tnq.contract_sliced_noalloc(state["plan"], state["bits"], *span, per_slice=case["per_slice"])
        else:
            out = tnq.contract_sliced(state["plan"], state["bits"], *span, workspace=state["workspace"],
                                      max_batch=state["batch"], per_slice=case["per_slice"])
        return _single(np.append(out[1], out[0])) if case["per_slice"] else _single(out)
    if kind == "serve":
        amps = tnq.amplitudes_batch(state["plans"], state["bits"], workspace=state["workspace"])
        n = state["each"]
        return [_single(amps[i * n:(i + 1) * n]) for i in range(len(state["plans"]))]
    if kind == "lattice":
        value, slices = tnq.contract_sliced(state["plan"], None, 0, state["end"], workspace=state["workspace"],
                                            per_slice=True)
        return _single(np.append(slices, value))
    case = state["case"]
    if kind == "train":
        weights, losses = learned.train(state["X"], state["y"], epochs=case["epochs"], batch=case["batch"], lr=0.02,
                                        mu=0.9, seed=state["seed"], hidden=case["hidden"])
        return {"weights": weights, "losses": np.asarray(losses, np.float32)}
    loss, grads = learned.gpu_grad(state["params"], state["X"], state["y"], case["hidden"])
    return {"loss": loss, "grads": grads}


# ---- the least work -------------------------------------------------------------
def _plan_work(plan, items):
    return dict(bytes=2.0 * 8 * 4 * plan.info()["n_leaf_tensors"] + 16.0 * items,
                flops=plan.info()["flops_per_slice"] * items)


def work(case):
    """Contractions: gate tensors in, values out; the additions and
    multiplications of bucket elimination in the plan's order (Eq. 2)."""
    kind = case["kind"]
    if kind == "amplitude":
        plan = _plan(case, _circuit(case))
        begin, end = _range(case, plan)
        return _plan_work(plan, end - begin)
    if kind == "serve":
        got = dict(bytes=0.0, flops=0.0)
        for c in _serve_circuits(case):
            plan = tnq.Plan(c, max_bag_log2=case["max_bag"], max_p=case["max_p"], reorder_every=case["reorder"],
                            precision=PRECISIONS[case["precision"]])
            w = _plan_work(plan, case["bitstrings"] * plan.info()["n_slices"])
            got = {k: got[k] + w[k] for k in got}
        return got
    if kind == "lattice":
        net = _network(case, 0)
        plan = _network_plan(case, net)
        w = _plan_work(plan, plan.info()["n_slices"])
        return dict(w, bytes=sum(16.0 * t.size for _, t in net.tensors) + 16.0 * plan.info()["n_slices"])
    F, H, rows = learned.features(), case["hidden"], case["rows"]
    weights = H * F + H + H * H + H + H + 1
    forward = 2.0 * (H * F + H * H + H)
    flops = forward + 2.0 * (H * F + 2 * H * H + 2 * H)  # a row's share of every gradient
    if kind == "train":
        steps = rows // min(case["batch"], rows) * case["epochs"]
        return dict(bytes=4.0 * (rows * (F + 1) + 2 * weights), flops=flops * steps * min(case["batch"], rows))
    return dict(bytes=4.0 * (rows * (F + 1) + 2 * weights), flops=flops * rows)


# ---- the same values in 64 bits, from plain torch --------------------------------
_R = 2.0 ** -0.5
_GATES = {inputs.H: [[_R, _R], [_R, -_R]], inputs.X_1_2: [[_R, -1j * _R], [-1j * _R, _R]],
          inputs.Y_1_2: [[_R, -_R], [_R, _R]]}


def _circuit_tensors(circ, bits):
    """(tensors, sizes): tensors as (variables, complex128 array); variable
    (q, k) is the value of qubit q's wire after k non-diagonal gates."""
    at = [0] * circ.n_qubits
    tensors = []
    for g in circ.gates:
        a = (g.q0, at[g.q0])
        if g.kind == inputs.T:
            tensors.append(([a], np.array([1, np.exp(0.25j * np.pi)])))
        elif g.kind == inputs.CZ:
            tensors.append(([a, (g.q1, at[g.q1])], np.array([[1, 1], [1, -1]])))
        else:
            at[g.q0] += 1
            tensors.append(([(g.q0, at[g.q0]), a], np.array(_GATES[g.kind])))
    for q in range(circ.n_qubits):
        tensors.append(([(q, 0)], np.array([1, 0])))
        tensors.append(([(q, at[q])], np.array([1 - bits[q], bits[q]])))
    return tensors, {(q, k): 2 for q in range(circ.n_qubits) for k in range(at[q] + 1)}


def _eliminate(tensors, sizes, keep, order):
    """Sum over every variable, restricted to the values keep[v], of the product of the tensors."""
    where = {v: i for i, v in enumerate(order)}
    live = []
    for vs, t in tensors:
        for ax in reversed(range(len(vs))):  # a variable with one value left goes from the tensor at once
            if vs[ax] in keep:
                t = np.take(t, keep[vs[ax]][0] if len(keep[vs[ax]]) == 1 else keep[vs[ax]], axis=ax)
        vs = [v for v in vs if len(keep.get(v, "  ")) != 1]
        by = sorted(range(len(vs)), key=lambda ax: -where[vs[ax]])  # the next one to go varies fastest
        t = torch.from_numpy(np.ascontiguousarray(np.transpose(t, by)).astype(np.complex128)).cuda()
        live.append(([vs[ax] for ax in by], t))
    buckets = {v: [] for v in order}
    total = torch.ones((), dtype=torch.complex128, device="cuda")
    for vs, t in live:
        if vs:
            buckets[vs[-1]].append((vs, t))
        else:
            total = total * t
    for v in order:
        own = sorted(buckets.pop(v), key=lambda x: len(x[0]))
        if not own:  # a variable that no tensor has counts each of its values
            total = total * len(keep.get(v, range(sizes[v])))
            continue
        have, out = [], None
        for vs, t in own:
            both = sorted(set(have) | set(vs), key=lambda w: -where[w])
            n = {**dict(zip(vs, t.shape)), **({} if out is None else dict(zip(have, out.shape)))}
            t = t.reshape([n[w] if w in vs else 1 for w in both])
            out = t if out is None else out.reshape([n[w] if w in have else 1 for w in both]) * t
            have = both
        out = out.sum(-1)
        if len(have) > 1:
            buckets[have[-2]].append((have[:-1], out))
        else:
            total = total * out
    return complex(total)


def _order(plan, sizes):
    """Every variable once: the plan's order, with those that it has fixed (one value each) before it."""
    free = plan.order()
    return [v for v in sizes if v not in set(free)] + free


def _exact_slices(circ, bits, plan, begin, end):
    tensors, sizes = _circuit_tensors(circ, bits)
    last = {q: max(k for p, k in sizes if p == q) for q in range(circ.n_qubits)}
    mu = plan.sliced()  # which variable is which bit of a slice's number
    order = _order(plan, sizes)
    got = []
    for s in range(begin, end):
        keep = {(q, 0): [0] for q in last}
        for q, k in last.items():  # a wire without a gate has one variable, both input and output
            keep[(q, k)] = [bits[q]] if k else [0]
        keep.update({v: [(s >> j) & 1] for j, v in enumerate(mu)})
        got.append(_eliminate(tensors, sizes, keep, order))
    return got


def _exact_lattice(case, seed):
    net = _network(case, seed)
    plan = _network_plan(case, net)
    sizes = dict(enumerate(net.dims))
    # an index goes when the last of its digits does
    last = {i: n for n, (i, digit) in enumerate(plan.order())}
    order = [i for i in sizes if i not in last] + sorted(last, key=lambda i: last[i])
    got = []
    for s in range(plan.info()["n_slices"]):
        keep = {}
        for j, (i, digit) in enumerate(plan.sliced()):
            keep[i] = [x for x in keep.get(i, range(sizes[i])) if (x >> digit) & 1 == (s >> j) & 1]
        got.append(_eliminate(net.tensors, sizes, keep, order))
    return _double(got + [sum(got)])


def _double(values):
    return np.asarray(values, np.complex128).reshape(-1)


def _mlp_grad(w, X, y):
    """Loss and gradients of mean((f(x) - y)^2) / 2 for the three-layer ReLU network, by torch in 64 bits."""
    w = [p.detach().requires_grad_() for p in w]
    h = torch.relu(X @ w[0].T + w[1])
    h = torch.relu(h @ w[2].T + w[3])
    loss = 0.5 * ((h @ w[4] + w[5] - y) ** 2).mean()
    return loss.detach(), torch.autograd.grad(loss, w)


def _split(flat, F, H):
    shapes = [(H, F), (H,), (H, H), (H,), (H,), (1,)]
    parts = torch.split(flat, [int(np.prod(s)) for s in shapes])
    return [p.reshape(s) for p, s in zip(parts, shapes)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "amplitude":
        circ = _circuit(case)
        plan = _plan(case, circ)
        begin, end = _range(case, plan)
        if plan.info()["flops_per_slice"] * (end - begin) > 1e12:
            return None
        got = _exact_slices(circ, inputs.random_bitstring(circ.n_qubits, seed), plan, begin, end)
        return _double(got + [sum(got)] if case["per_slice"] else [sum(got)])
    if kind == "serve":
        circuits = _serve_circuits(case)
        out = []
        for circ, bits in zip(circuits, _serve_bits(case, circuits, seed)):
            plan = tnq.Plan(circ, max_bag_log2=case["max_bag"], max_p=case["max_p"], reorder_every=case["reorder"])
            n = plan.info()["n_slices"]
            if len(circuits) * case["bitstrings"] * n > 100 or plan.info()["flops_per_slice"] > 1e10:
                out.append(None)
                continue
            out.append(_double([sum(_exact_slices(circ, b, plan, 0, n)) for b in bits]))
        return out if any(o is not None for o in out) else None
    if kind == "lattice":
        return _exact_lattice(case, seed)
    X, y = (torch.from_numpy(v).cuda().double() for v in _rows(case, seed))
    H, F = case["hidden"], X.shape[1]
    flat = torch.from_numpy(learned.init_params(seed, H)).cuda().double()
    if kind == "grad":
        loss, grads = _mlp_grad(_split(flat, F, H), X, y)
        return {"loss": loss.reshape(1), "grads": torch.cat([g.reshape(-1) for g in grads])}
    gen = torch.Generator(device="cpu").manual_seed(seed)
    batch = min(case["batch"], case["rows"])
    momentum, losses = torch.zeros_like(flat), []
    for _ in range(case["epochs"]):
        perm, total = torch.randperm(case["rows"], generator=gen).cuda(), 0.0
        for i in range(0, case["rows"] - batch + 1, batch):
            loss, grads = _mlp_grad(_split(flat, F, H), X[perm[i:i + batch]], y[perm[i:i + batch]])
            momentum = 0.9 * momentum + torch.cat([g.reshape(-1) for g in grads])
            flat = flat - 0.02 * momentum
            total += float(loss)
        losses.append(total / max(1, case["rows"] // batch))
    return {"weights": flat.cpu().numpy(), "losses": np.asarray(losses)}
