"""Pairwise contraction of fragment graphs that are no stars (needs a GPU).

The contraction order is planned from the fragment graph: chains from four
blocks to the twelve-cut limit, branched trees, a fragment graph with a cycle
and a double edge, cut-free fragments beside a chain (outer products), empty
and wide marginals, several problems of different depth in one plan.  Each is
compared with the definition itself (the sum over the cut index, which partial
ranges still use: two halves added) and with the uncut statevector where that
fits.

Tolerances: 1e-5, the parity bar, against the statevector; 2e-6 against the
direct sum, whose FP32 terms carry at most 13 roundings of 2^-24 each
(7.7e-7) on a sum of absolute terms of order one.
"""
import numpy as np
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import CX, CZ, H, S, T, Circuit, Workload, tree_circuit
from oracle.pipeline import brute_force

pytestmark = pytest.mark.gpu


def tree(parents, marg, zs=(), seed=1, n_t=3):
    c, cuts = tree_circuit(parents, 14, n_t, seed=seed)
    return Workload("tree", c, cuts, [q % c.n_qubits for q in marg], [list(z) for z in zs], 256, 3)


def ring():
    """Fragments A, B, C joined A-B twice, A-C and B-C: no fragment on every cut."""
    c = Circuit(8)
    for q in range(8):
        c.add(H, q)
    for q in (0, 1, 2, 4):
        c.add(S, q)
    cuts = []
    for a, b in ((0, 1), (1, 2), (2, 0)):
        c.add(CX, a, b)
    c.add(T, 1)
    for src, q in ((0, 3), (2, 7), (1, 5)):       # one gate with A, then the wire moves on
        c.add(CX, src, q)
        c.add(S, q)
        cuts.append((q, len(c.gates)))
    c.add(CZ, 3, 4)
    c.add(H, 3)
    c.add(CX, 7, 4)
    c.add(T, 4)
    c.add(CX, 4, 6)
    c.add(H, 6)
    cuts.append((6, len(c.gates)))
    c.add(CX, 5, 6)
    c.add(H, 5)
    c.add(CX, 6, 5)
    return Workload("ring", c, cuts, [6, 0, 3, 5, 7], [[0, 6], [3, 5, 7], [1]], 256, 3)


def with_idle(parents, marg):
    """A chain beside qubits of their own: fragments without any cut."""
    w = tree(parents, marg, seed=4)
    n = w.circuit.n_qubits
    c = Circuit(n + 2)
    c.gates = list(w.circuit.gates) + [(H, n, -1), (H, n + 1, -1), (T, n + 1, -1), (H, n + 1, -1)]
    return Workload("idle", c, w.cuts, w.marginal + [n + 1, n], [[0, n + 1], [n]], 256, 3)


CASES = {
    "chain4": lambda: [tree([0, 1, 2], [0, 5, 11, 7], [[0, 1], [11]])],
    "chain5_wide": lambda: [tree([0, 1, 2, 3], list(range(14)), [[3, 12]])],
    "chain6_empty": lambda: [tree([0, 1, 2, 3, 4], [], [[0], [17, 2]])],
    "chain12": lambda: [tree(list(range(11)), [0, 20, 35], [[0, 35], [1, 2]], seed=2)],
    "branches": lambda: [tree([0, 0, 0, 1, 1, 2], [1, 4, 9, 20, 13], [[2, 20]])],
    "ring": lambda: [ring()],
    "idle": lambda: [with_idle([0, 1, 2], [0, 3, 10])],
    "several": lambda: [tree([0, 1, 2], [0, 5]), tree(list(range(8)), [2, 20, 9], [[1, 2]]), ring(),
                        tree([0, 0, 1], [1, 11, 4, 6])],
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("mode", [ccs.CCS_EXACT, ccs.CCS_SAMPLED], ids=["exact", "sampled"])
def test_pairwise_equals_direct_sum(name, mode):
    ws = CASES[name]()
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, ws)
    for pi, w in enumerate(ws):
        nf, k = ccs.ccs_plan_counts(ctx, plan, pi)
        slots = [ccs.ccs_fragment_info_get(ctx, plan, pi, f)["n_slots"] for f in range(nf)]
        assert max(slots) < k, "a star"
    res = ccs.ccs_eval_variants(ctx, plan, mode=mode, shots=300)
    m, z = ccs.ccs_recombine(ctx, plan, res)
    kmax = max(len(w.cuts) for w in ws)
    halves = [ccs.ccs_recombine(ctx, plan, res, k_range=r) for r in ((0, 4 ** kmax // 2), (4 ** kmax // 2, 0))]
    assert np.abs(m - halves[0][0] - halves[1][0]).max() < 2e-6
    if len(z):
        assert np.abs(z - halves[0][1] - halves[1][1]).max() < 2e-6
    for graph in (False, True):
        mb, _ = ccs.ccs_recombine(ctx, plan, res, precision=ccs.CCS_BF16, use_graph=graph)
        assert np.abs(mb - m).max() < 1e-2
    if mode == ccs.CCS_EXACT and max(w.circuit.n_qubits for w in ws) <= 20:
        exact = [brute_force(w.circuit, w.marginal, w.zstrings) for w in ws]
        assert np.abs(m - np.concatenate([e[0] for e in exact])).max() < 1e-5
        if len(z):
            assert np.abs(z - np.concatenate([e[1] for e in exact])).max() < 1e-5
