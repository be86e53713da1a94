"""Timed cases of the circuit-cutting path: the work a program has the library do.

Every case is one pass through the public entry points of
``paper_2303_10788_gb300.ccs``: evaluate a plan's variants and recombine them
(optionally with the maximum-likelihood correction between), a whole call from
host circuits to host results, or one gradient / one prediction of the cut
scorer.  ``prepare`` makes what the program holds before the pass (circuits
drawn from the seed, the plan, the result buffers); ``run`` is the pass.

The library computes probabilities in FP32 and hands them out as doubles; the
programs here keep them in single precision, so ``run`` returns float32.
"""
from types import SimpleNamespace

import numpy as np
import torch

from paper_2303_10788_gb300 import ccs

H, S, SDG, X, Y, Z, CX, CZ, T, TDG = range(10)
_F32 = torch.float32


# --- the cases -----------------------------------------------------------------

def listed():
    return [
        # one small near-Clifford circuit, results wanted on the host at once: the
        # smallest call a user makes, default options (latency and launches)
        _star("star16", n=16, depth=12, regions=1, width=5, n_t=2, marginal=8, zstrings=16, shots=4096, host=True),
        # the largest QAOA instance of the method's evaluation, strong simulation, cuts searched
        dict(name="qaoa26", kind="qaoa", n=26, rounds=1, circuits=1, marginal=10, zstrings=8, shots=0, mode="exact",
             graph=True, tune=False),
        # one 100-qubit circuit with two wide non-Clifford regions and 64 observables
        _star("star100", n=100, depth=20, regions=2, width=8, n_t=10, marginal=12, zstrings=64, shots=10000),
        # the largest single circuit: 20736 variants of a 500-wire body, 4^8 cut terms
        _star("star500", n=500, depth=30, regions=4, width=1, n_t=16, marginal=16, zstrings=0, shots=16384),
        # a wide contraction in BF16 (tensor cores): 4^8 cut terms, 2^9 hub outputs, an odd qubit count
        _star("star301_bf16", n=301, depth=24, regions=4, width=2, n_t=9, marginal=13, zstrings=0, shots=4096,
              precision="bf16"),
        # a VQE sweep: many deep, narrow circuits in one plan, cuts searched, launch shapes tuned
        dict(name="vqe300x64", kind="vqe", n=300, rounds=5, circuits=64, marginal=10, zstrings=8, shots=5000,
             mode="sampled", graph=True, tune=True),
        # many different circuits in one plan (throughput serving)
        _batch("batch64", circuits=64, shots=4096, tune=True),
        # a smaller batch whose sampled fragment models are corrected by maximum likelihood
        _batch("batch16_ml", circuits=16, shots=4096, ml=True),
        # strong simulation of a batch (no shots, the Clifford-specific stitching)
        _batch("batch32_stitch", circuits=32, shots=0, mode="stitch"),
        # fragments in a chain: nine blocks, eight cuts, no fragment on every cut
        dict(name="chain9", kind="tree", blocks=9, chain=True, gates=24, n_t=4, marginal=10, zstrings=8, shots=0,
             mode="exact", graph=False, host=False),
        # one minibatch of training the cut scorer: loss and gradient
        dict(name="scorer_grad64", kind="scorer", graphs=64, n_lo=50, n_hi=400, train=True),
        # a request served from host circuits to host results, plan build included
        _batch("serve16", circuits=16, shots=4096, serve=True, graph=False),
    ]


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["star", "star", "star", "batch", "batch", "serve", "ml", "vqe", "qaoa", "tree", "scorer"])
    if kind == "star":
        regions = rng.choice([1, 2, 2, 3, 3, 4])
        width = rng.randint(1, 8) if regions < 4 else rng.randint(1, 3)
        n = max(_log_int(rng, 16, 500), regions * (width + 3) + 8)
        mode = rng.choice(["sampled", "sampled", "sampled", "stitch", "exact"]) if regions < 4 else "sampled"
        hi = 16 if mode == "sampled" else 13
        marginal = rng.randint(regions + 2, min(hi, n - regions * width + regions))
        return _star(None, n=n, depth=rng.randint(8, 30), regions=regions, width=width,
                     n_t=regions * rng.randint(1, 4), marginal=marginal, zstrings=rng.choice([0, 0, 1, 8, 33, 64]),
                     shots=_log_int(rng, 500, 16384) if mode == "sampled" else 0, mode=mode,
                     precision=rng.choice(["fp32", "fp32", "bf16"]), host=rng.random() < 0.3,
                     graph=rng.random() < 0.6)
    if kind == "batch":
        mode = rng.choice(["sampled", "sampled", "stitch"])
        return _batch(None, circuits=_log_int(rng, 2, 64), shots=_log_int(rng, 500, 8192) if mode == "sampled" else 0,
                      mode=mode, graph=rng.random() < 0.7)
    if kind == "serve":
        return _batch(None, circuits=_log_int(rng, 1, 16), shots=_log_int(rng, 500, 8192), serve=True, graph=False)
    if kind == "ml":
        return _batch(None, circuits=_log_int(rng, 1, 16), shots=_log_int(rng, 500, 8192), ml=True)
    if kind == "vqe":
        return dict(kind="vqe", n=_log_int(rng, 20, 300), rounds=rng.randint(1, 5), circuits=_log_int(rng, 1, 64),
                    marginal=rng.randint(4, 10), zstrings=rng.choice([0, 3, 8]), shots=_log_int(rng, 500, 8192),
                    mode="sampled", graph=rng.random() < 0.7, tune=False)
    if kind == "qaoa":
        mode = rng.choice(["exact", "sampled"])
        return dict(kind="qaoa", n=rng.randint(8, 26), rounds=rng.randint(1, 2), circuits=rng.randint(1, 4),
                    marginal=rng.randint(3, 8), zstrings=rng.choice([0, 5, 8]),
                    shots=_log_int(rng, 500, 8192) if mode == "sampled" else 0, mode=mode, graph=rng.random() < 0.5,
                    tune=False)
    if kind == "tree":
        mode = rng.choice(["exact", "sampled"])
        blocks = rng.randint(4, 9)
        return dict(kind="tree", blocks=blocks, chain=rng.random() < 0.5, gates=rng.randint(8, 30),
                    n_t=rng.randint(1, 5), marginal=rng.randint(3, 10), zstrings=rng.choice([0, 4, 8]),
                    shots=_log_int(rng, 500, 8192) if mode == "sampled" else 0, mode=mode, graph=rng.random() < 0.5,
                    host=rng.random() < 0.5)
    return dict(kind="scorer", graphs=_log_int(rng, 1, 64), n_lo=rng.randint(10, 100), n_hi=rng.randint(101, 400),
                train=rng.random() < 0.5)


def _log_int(rng, lo, hi):
    return min(hi, int(round(lo * (hi / lo) ** rng.random())))


def _star(name, **kw):
    c = dict(kind="star", n=0, depth=0, regions=1, width=1, n_t=1, marginal=8, zstrings=0, shots=4096, mode="sampled",
             precision="fp32", host=False, graph=True)
    c.update(kw)
    if c["host"]:
        c["graph"] = False
    return dict(name=name, **c) if name else c


def _batch(name, **kw):
    c = dict(kind="batch", circuits=1, shots=4096, mode="sampled", ml=False, serve=False, graph=True, tune=False)
    c.update(kw)
    return dict(name=name, **c) if name else c


# --- circuits --------------------------------------------------------------------

def _table(words, width):
    t = np.full((len(words), width), -1, np.int64)
    for i, w in enumerate(words):
        t[i, :len(w)] = w
    return t


# the 24 one-qubit Cliffords as gate words, and R_y / R_z / R_x of multiples of pi/2
_C1 = _table([p + q for p in ([], [H], [S], [H, S, H], [H, S], [S, H]) for q in ([], [X], [Y], [Z])], 4)
_RZ = _table([[], [S], [Z], [SDG]], 1)
_RY = _table([[], [Z, H], [Y], [H, Z]], 2)
_RX = _table([[], [H, S, H], [X], [H, SDG, H]], 3)


def _one_qubit(words, q):
    """Gate slots [len(q), width, 3] of one word per qubit; an absent gate has op -1."""
    g = np.full(words.shape + (3,), -1, np.int64)
    g[..., 0] = words
    g[..., 1] = np.asarray(q)[:, None]
    return g


def _flat(slots):
    g = slots.reshape(-1, 3)
    return g[g[:, 0] >= 0]


def _layer(rng, pairs):
    """A random two-qubit Clifford on every pair: local words, one to three CX, local words."""
    a, b = pairs[:, 0], pairs[:, 1]
    k = len(pairs)
    words = _C1[rng.integers(24, size=(4, k))]
    n_cx = rng.choice([1, 2, 3], size=k, p=[0.47, 0.47, 0.06])
    core = np.full((k, 3, 3), -1, np.int64)
    for i in range(3):
        on = n_cx > i
        core[on, i, 0] = CX
        core[:, i, 1], core[:, i, 2] = (a, b) if i % 2 == 0 else (b, a)
    return _flat(np.concatenate([_one_qubit(words[0], a), _one_qubit(words[1], b), core, _one_qubit(words[2], a),
                                 _one_qubit(words[3], b)], axis=1))


def _star_circuit(rng, n, depth, widths, n_t, marginal):
    """Brickwork whose non-Clifford regions (some full qubits and a time window
    of the next qubit) are joined to the Clifford body by two cut wires each."""
    gap = (n - sum(widths) - len(widths)) // (len(widths) + 1)
    regs, at = [], gap // 2
    for w in widths:
        ta = int(rng.integers(2, max(3, depth // 2)))
        tb = int(min(depth - 2, ta + 2 + rng.integers(0, max(1, depth // 2))))
        regs.append((at, w, min(ta, tb - 2), tb))
        at += w + 1 + gap
    t_slots = {}
    for i, (s, w, _, _) in enumerate(regs):
        for _ in range(max(1, n_t // len(regs))):
            t_slots.setdefault(int(rng.integers(depth)), []).append(s + int(rng.integers(w)))
    gates, cuts, count = [], [], 0
    for layer in range(depth):
        frag = np.zeros(n, np.int64)
        for i, (s, w, ta, tb) in enumerate(regs):
            frag[s:s + w] = i + 1
            if ta <= layer < tb:
                frag[s + w] = i + 1
            if layer in (ta, tb):
                cuts.append((s + w, count))
        pairs = []
        for f in range(len(regs) + 1):
            members = np.flatnonzero(frag == f)[layer % 2:]
            members = members[:len(members) // 2 * 2]
            pairs.append(members.reshape(-1, 2))
        pairs = np.concatenate(pairs)
        g = _layer(rng, pairs[np.argsort(pairs[:, 0], kind="stable")])
        if layer in t_slots:
            g = np.concatenate([g, [(T, q, -1) for q in sorted(set(t_slots[layer]))]])
        gates.append(g)
        count += len(g)
    inside = np.concatenate([np.arange(s, s + w) for s, w, _, _ in regs])
    body = np.setdiff1d(np.arange(n), inside)
    marg = [s for s, _, _, _ in regs]
    marg += sorted(int(q) for q in rng.choice(body, size=marginal - len(regs), replace=False))
    return np.concatenate(gates), cuts, marg


def _batch_circuit(rng):
    """50-300 qubits, depth 10-40, one to three regions, 2-12 T, a 10-qubit marginal."""
    n, depth, regions = int(rng.integers(50, 301)), int(rng.integers(10, 41)), int(rng.integers(1, 4))
    widths = [int(rng.integers(1, 10)) for _ in range(regions)]
    return (n,) + _star_circuit(rng, n, depth, widths, int(rng.integers(2, 13)), 10)


def _with_t(rng, gates, n):
    """One T or its inverse at a random place."""
    at = int(rng.integers(len(gates) + 1))
    return np.insert(gates, at, [T if rng.random() < 0.5 else TDG, int(rng.integers(n)), -1], axis=0)


def _vqe_circuit(rng, n, rounds):
    """Hardware-efficient ansatz at Clifford angles: rotations, a CX chain, rotations."""
    q = np.arange(n)
    chain = np.stack([np.full(n - 1, CX), q[:-1], q[1:]], axis=1)

    def rotations():
        return _flat(np.concatenate([_one_qubit(_RY[rng.integers(4, size=n)], q),
                                     _one_qubit(_RZ[rng.integers(4, size=n)], q)], axis=1))
    parts = []
    for _ in range(rounds):
        parts += [rotations(), chain, rotations()]
    return _with_t(rng, np.concatenate(parts), n)


def _qaoa_circuit(rng, n, rounds):
    """MaxCut on the Sherrington-Kirkpatrick model at Clifford angles: every pair, then the mixer."""
    q = np.arange(n)
    parts = [np.stack([np.full(n, H), q, np.full(n, -1)], axis=1)]
    a, b = np.triu_indices(n, 1)
    for _ in range(rounds):
        g, m = int(rng.integers(1, 4)), int(rng.integers(1, 4))
        word = _RZ[(g * rng.choice([1, 3], size=len(a))) % 4]
        cx = np.stack([np.full(len(a), CX), a, b], axis=1)[:, None, :]
        parts.append(_flat(np.concatenate([cx, _one_qubit(word, b), cx], axis=1)))
        parts.append(_flat(_one_qubit(np.tile(_RX[m], (n, 1)), q)))
    return _with_t(rng, np.concatenate(parts), n)


def _tree_circuit(rng, blocks, chain, per_block, n_t):
    """Blocks of three wires joined in a chain or a tree by one cut CX each."""
    n = 3 * blocks
    parents = [b - 1 if chain else int(rng.integers(b)) for b in range(1, blocks)]
    gates = [(H, q, -1) for q in range(n)]

    def fill(before):
        for _ in range(per_block * blocks // 2):
            b = int(rng.integers(blocks))
            qs = [3 * b, 3 * b + 1, 3 * b + 2]
            if rng.random() < 0.45:
                u, v = rng.choice(qs[1:] if before and b else qs, size=2, replace=False)
                gates.append((CX if rng.random() < 0.5 else CZ, int(u), int(v)))
            else:
                gates.append((int(rng.integers(6)), int(rng.choice(qs)), -1))
    fill(True)
    gates += [(CX, 3 * p + 1, 3 * b) for b, p in enumerate(parents, start=1)]
    cuts = [(3 * b, len(gates)) for b in range(1, blocks)]
    for b in range(blocks):                       # each block is one fragment after its cut
        gates += [(CX, 3 * b, 3 * b + 1), (CX, 3 * b + 1, 3 * b + 2)]
    start = len(gates)
    fill(False)
    for _ in range(n_t):
        gates.insert(int(rng.integers(start, len(gates) + 1)), (T, int(rng.integers(n)), -1))
    return np.asarray(gates, np.int64), cuts


def _problems(case, seed):
    """The case's circuits: (n, gates, cuts or None, marginal, zstrings) each."""
    rng = np.random.default_rng([seed, 2303])
    out = []
    for _ in range(case.get("circuits", 1)):
        if case["kind"] == "batch":
            n, gates, cuts, marg = _batch_circuit(rng)
        elif case["kind"] == "star":
            n = case["n"]
            gates, cuts, marg = _star_circuit(rng, n, case["depth"], [case["width"]] * case["regions"], case["n_t"],
                                              case["marginal"])
        else:
            if case["kind"] == "tree":
                n = 3 * case["blocks"]
                gates, cuts = _tree_circuit(rng, case["blocks"], case["chain"], case["gates"], case["n_t"])
            else:
                n, cuts = case["n"], None
                make = _vqe_circuit if case["kind"] == "vqe" else _qaoa_circuit
                gates = make(rng, n, case["rounds"])
            marg = sorted(int(q) for q in rng.choice(n, size=case["marginal"], replace=False))
        zs = [sorted(int(q) for q in rng.choice(n, size=int(rng.integers(1, min(n, 8) + 1)), replace=False))
              for _ in range(case.get("zstrings", 0))]
        out.append((n, gates, cuts, marg, zs))
    return out


# --- prepare and run ---------------------------------------------------------------

_MODES = {"exact": ccs.CCS_EXACT, "sampled": ccs.CCS_SAMPLED, "stitch": ccs.CCS_STITCH}


def prepare(case, seed):
    if case["kind"] == "scorer":
        return _prepare_scorer(case, seed)
    probs = []
    for n, gates, cuts, marg, zs in _problems(case, seed):
        probs.append(SimpleNamespace(circuit=SimpleNamespace(n_qubits=n, gates=gates.tolist()), cuts=cuts,
                                     marginal=marg, zstrings=zs))
    packed = ccs.pack_problems(probs)
    for p in probs:                 # marshalled: the gate lists are no longer needed
        p.circuit.gates = None
    serve = case.get("serve", False)
    st = SimpleNamespace(case=case, serve=serve, packed=packed, ctx=ccs.ccs_create(0, torch_allocator=not serve))
    mode = case["mode"]
    st.ev = dict(mode=_MODES[mode], shots=case["shots"] if mode == "sampled" else 1024,
                 seed_lo=(seed * 2654435761) & 0xffffffff, seed_hi=seed & 0x7fffffff)
    st.precision = ccs.CCS_BF16 if case.get("precision") == "bf16" else ccs.CCS_FP32
    st.graph, st.ml, st.host = case["graph"], case.get("ml", False), case.get("host", False) or serve
    st.plan = st.res = None
    if serve:
        return st
    st.plan = ccs.ccs_build_fragments(st.ctx, packed)
    # the result's buffers (and tuned launch shapes) the program keeps for this plan
    st.res = ccs.ccs_eval_variants(st.ctx, st.plan, autotune=case.get("tune", False), **st.ev)
    if not st.host:
        st.marg = torch.empty(sum(1 << len(p.marginal) for p in probs), dtype=torch.float64, device="cuda")
        st.zexp = torch.empty(max(1, sum(len(p.zstrings) for p in probs)), dtype=torch.float64, device="cuda")
    st.n_z = sum(len(p.zstrings) for p in probs)
    return st


def run(st):
    if st.case["kind"] == "scorer":
        return _run_scorer(st)
    plan, res = st.plan, st.res
    if st.serve:
        plan = ccs.ccs_build_fragments(st.ctx, st.packed)
    res = ccs.ccs_eval_variants(st.ctx, plan, use_graph=st.graph, res=res, **st.ev)
    if st.ml:
        ccs.ccs_ml_correct(st.ctx, plan, res)
    if st.host:
        marg, zexp = ccs.ccs_recombine(st.ctx, plan, res, precision=st.precision)
        return {"marginal": marg.astype(np.float32), "zexp": zexp.astype(np.float32)}
    ccs.ccs_recombine(st.ctx, plan, res, precision=st.precision, marginal_out=st.marg, zexp_out=st.zexp,
                      use_graph=st.graph)
    out = {"marginal": st.marg.to(_F32)}
    if st.n_z:
        out["zexp"] = st.zexp.to(_F32)
    return out


# --- the cut scorer ------------------------------------------------------------------

_HID, _LAYERS = 64, 3


def _scorer_graphs(case, seed):
    """Graphs of brickwork circuits as the featuriser makes them: a chain of
    interacting qubits (gate counts as weights, rows of A normalised), eight
    node features and eight global ones."""
    rng = np.random.default_rng([seed, 1078])
    graphs = []
    for _ in range(case["graphs"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        w = rng.integers(3, 30, size=n - 1).astype(np.float64)
        left, right = np.concatenate([[0.0], w]), np.concatenate([w, [0.0]])
        deg = left + right
        row = np.repeat(np.arange(n), 2)
        col = np.stack([np.arange(n) - 1, np.arange(n) + 1], axis=1).ravel()
        wt = np.stack([left, right], axis=1).ravel()
        keep = wt > 0
        row, col, wt = row[keep], col[keep], wt[keep]
        x = np.zeros((n, 8), np.float32)
        x[:, 0] = 1.0
        x[:, 1] = rng.poisson(0.1, n) / 4.0
        x[:, 2] = np.bincount(row, minlength=n) / 4.0
        x[:, 3] = rng.integers(40, 300, n) / 100.0
        x[:, 4] = (rng.random(n) < 0.05) * rng.random(n)
        x[:, 5] = (rng.random(n) < 0.03) * 2.0
        x[:, 6] = rng.random(n) < 10.0 / n
        x[:, 7] = rng.random(n) < 0.9
        glob = np.array([rng.integers(2, 9) / 8.0, rng.random(), rng.random(), rng.random(), rng.random(),
                         np.log2(n) / 9.0, rng.uniform(0.6, 1.0), rng.integers(2, 6) / 8.0], np.float32)
        rowptr = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=n))]).astype(np.int32)
        graphs.append(ccs.Graph(x, rowptr, col.astype(np.int32), (wt / deg[row]).astype(np.float32),
                                (wt / deg[col]).astype(np.float32), glob))
    params = []
    for rows, cols in [(_HID, 8)] + [(_HID, _HID)] * (2 * _LAYERS) + [(_HID, _HID + 8), (1, _HID)]:
        params.append(rng.uniform(-1, 1, (rows, cols)) * np.sqrt(6.0 / cols) * 0.7)
    bias = [rng.normal(0, 0.05, k) for k in (_HID, _HID, _HID, _HID, _HID, 1)]
    order = [params[0], bias[0]]
    for l in range(_LAYERS):
        order += [params[1 + 2 * l], params[2 + 2 * l], bias[1 + l]]
    order += [params[7], bias[4], params[8], bias[5]]
    theta = np.concatenate([np.ravel(p) for p in order]).astype(np.float32)
    target = rng.normal(0.0, 1.0, case["graphs"]).astype(np.float32)
    return graphs, theta, target


def _prepare_scorer(case, seed):
    graphs, theta, target = _scorer_graphs(case, seed)
    st = SimpleNamespace(case=case, ctx=ccs.ccs_create(0), batch=ccs.make_batch(graphs), target=target)
    st.net = ccs.ccs_mpnn_create(st.ctx)
    ccs.ccs_mpnn_set_params(st.ctx, st.net, theta)
    return st


def _run_scorer(st):
    if st.case["train"]:
        loss, grad = ccs.ccs_mpnn_gradient(st.ctx, st.net, st.batch, st.target)
        return {"loss": np.float32(loss), "grad": grad}
    return {"pred": ccs.ccs_mpnn_forward(st.ctx, st.net, st.batch)}


# --- 64-bit results --------------------------------------------------------------------

def exact(case, seed):
    """The same results in 64 bits, without the library: a dense statevector of
    the uncut circuit (strong simulation of up to 27 qubits), the scorer's
    network and its gradient.  Sampled results have no such value, and larger
    circuits are out of a statevector's reach."""
    if case["kind"] == "scorer":
        return _exact_scorer(case, seed)
    probs = _problems(case, seed) if case["kind"] in ("star", "qaoa", "tree") and case["mode"] != "sampled" else []
    if not probs or case.get("precision") == "bf16" or max(p[0] for p in probs) > 27:
        return None
    marg, zexp = [], []
    for n, gates, _, m, zs in probs:
        p, z = _statevector(n, gates, m, zs)
        marg.append(p)
        zexp += z
    host = case.get("host", False)
    out = {"marginal": np.concatenate(marg)}
    if host or zexp:
        out["zexp"] = np.asarray(zexp, np.float64)
    return out


def _statevector(n, gates, marginal, zstrings):
    r = 0.5 ** 0.5
    one = {H: [[r, r], [r, -r]], X: [[0, 1], [1, 0]], Y: [[0, -1j], [1j, 0]]}
    phase = {S: 1j, SDG: -1j, Z: -1, T: complex(r, r), TDG: complex(r, -r)}
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1
    for op, a, b in gates.tolist():               # qubit q is bit q of the index
        v = psi.view(1 << (n - 1 - a), 2, 1 << a)
        if op in phase:
            v[:, 1] *= phase[op]
        elif op in one:
            u = one[op]
            lo, hi = v[:, 0].clone(), v[:, 1].clone()
            v[:, 0] = u[0][0] * lo + u[0][1] * hi
            v[:, 1] = u[1][0] * lo + u[1][1] * hi
        else:
            h, l = max(a, b), min(a, b)
            w = psi.view(1 << (n - 1 - h), 2, 1 << (h - l - 1), 2, 1 << l)
            if op == CZ:
                w[:, 1, :, 1] *= -1
            else:
                lo = w[:, 1, :, 0] if a == h else w[:, 0, :, 1]
                hi = w[:, 1, :, 1]
                t = lo.clone()
                lo.copy_(hi)
                hi.copy_(t)
    p = psi.real ** 2 + psi.imag ** 2
    z = []
    for qs in zstrings:
        f = p
        for q in sorted(qs):                       # removing low qubits first shifts the others down
            at = q - sum(1 for x in qs if x < q)
            g = f.view(-1, 2, 1 << at)
            f = (g[:, 0] - g[:, 1]).reshape(-1)
        z.append(float(f.sum()))
    keep = sorted(marginal)
    f = p.view([2] * n)                            # dimension n-1-q is qubit q
    f = f.sum(dim=[n - 1 - q for q in range(n) if q not in keep]) if len(keep) < n else f
    m = len(keep)
    f = f.permute([m - 1 - keep.index(marginal[m - 1 - i]) for i in range(m)])
    return f.reshape(-1).cpu().numpy(), z


def _exact_scorer(case, seed):
    graphs, theta, target = _scorer_graphs(case, seed)
    th = torch.from_numpy(theta).half().double().requires_grad_(True)       # weights are used in FP16
    at = [0]

    def take(*shape):
        k = int(np.prod(shape))
        at[0] += k
        return th[at[0] - k:at[0]].view(*shape)
    w_in, b_in = take(_HID, 8), take(_HID)
    layers = [(take(_HID, _HID), take(_HID, _HID), take(_HID)) for _ in range(_LAYERS)]
    w1, b1, w2, b2 = take(_HID, _HID + 8), take(_HID), take(_HID), take(1)
    pred = []
    for g in graphs:
        n = g.x.shape[0]
        a = torch.sparse_csr_tensor(torch.from_numpy(g.rowptr.astype(np.int64)), torch.from_numpy(g.col.astype(np.int64)),
                                    torch.from_numpy(g.val).double(), size=(n, n)).to_dense()
        h = torch.relu(torch.from_numpy(g.x).double() @ w_in.T + b_in)
        for ws, wn, b in layers:
            h = torch.relu(h @ ws.T + (a @ h) @ wn.T + b)
        r = torch.cat([h.mean(dim=0), torch.from_numpy(g.glob).double()])
        pred.append(torch.relu(w1 @ r + b1) @ w2 + b2[0])
    pred = torch.stack(pred)
    if not case["train"]:
        return {"pred": pred.detach().numpy()}
    loss = ((pred - torch.from_numpy(target).double()) ** 2).mean()
    loss.backward()
    return {"loss": loss.item(), "grad": th.grad.numpy()}


# --- work ------------------------------------------------------------------------------

def work(case):
    """Bytes a pass cannot do without (the circuits' gates as the library's
    8-byte fused two-qubit updates, or as given where they come from the host;
    the results once) and its operations (shots: the generator's rounds and the
    counting; the contraction leaf by leaf; the correction's eigenproblems)."""
    if case["kind"] == "scorer":
        nodes = case["graphs"] * (case["n_lo"] + case["n_hi"]) / 2.0
        mul = nodes * (8 * _HID + 2 * _LAYERS * _HID * _HID + 3 * _LAYERS * _HID)
        return {"bytes": nodes * (8 * 4 + 3 * 12 + 8) + 4 * 30000, "flops": 2 * mul * (3 if case["train"] else 1)}
    circuits = case.get("circuits", 1)
    if case["kind"] == "tree":
        k, m = case["blocks"] - 1, case["marginal"]
        ops = 12 * 40.0 * case["blocks"] * case["gates"] + 2.0 * 16 * (1 << m) * k
        ops += 12.0 * case["blocks"] * case["shots"] * 14
        return {"bytes": 8.0 * case["blocks"] * case["gates"] + 4.0 * (1 << m), "flops": ops}
    if case["kind"] == "batch":
        shapes, n, depth, m, gates = [(r, 1.0 / 3) for r in (1, 2, 3)], 175, 25, 10, 23000
    elif case["kind"] == "star":
        shapes, n, depth, m = [(case["regions"], 1.0)], case["n"], case["depth"], case["marginal"]
        gates = 10 * n * depth / 2
    else:
        shapes, n, depth, m = [(1, 1.0)], case["n"], 4 * case["rounds"], case["marginal"]
        depth = depth if case["kind"] == "vqe" else case["rounds"] * n
        gates = 10 * n * depth / 2
    rows = 24.0 * gates if case.get("serve") else 8.0 * n * depth / 2
    ops = 4.0 * n * n * depth / 64
    for r, share in shapes:
        per_word = 4 if m <= 8 else 2
        hub = 1 << max(0, m - r)
        ops += share * 12 ** r * case["shots"] * (40.0 / (4 * per_word) + 4)
        ops += share * sum(2.0 * hub * 16 ** r * 2 ** l / 16 ** (l - 1) for l in range(1, r + 1))
        if case.get("ml"):
            ops += share * hub * 8.0 * 9 * (1 << (2 * r)) ** 3
    return {"bytes": circuits * (rows + 4.0 * ((1 << m) + case.get("zstrings", 0))), "flops": circuits * ops}
