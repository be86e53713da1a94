"""Fragment graphs with many cuts between two fragments (needs a GPU).

Contracting such a pair sums 4^cuts terms for few entries, and several threads
share one entry: up to a warp, more than a warp, a whole CTA.  Cases: two
fragments joined by two to six cuts beside another pair, a triangle with one
such edge, both in one plan, no or several marginal bits, Z-strings.  Compared
with the definition itself (partial ranges sum the whole cut index; two halves
added) and with the uncut statevector.

Tolerances: 1e-5, the parity bar, against the statevector; 2e-6 against the
direct sum, whose FP32 terms carry at most 13 roundings of 2^-24 each on a sum
of absolute terms of order one.
"""
import numpy as np
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import CX, CZ, H, S, T, Circuit, Workload
from oracle.pipeline import brute_force

pytestmark = pytest.mark.gpu


def mixer(c, qs):
    for layer in range(2):
        for i, q in enumerate(qs):
            c.add(H, q)
            c.add(S, qs[(i + layer) % len(qs)])
            if len(qs) > 1:
                c.add(CX if (i + layer) % 2 else CZ, q, qs[(i + 1) % len(qs)])


def fat_edge(n, marginal_bits, triangle=False):
    """Fragments A and B joined by n cuts; C and D by one, or (triangle) C joined to
    A and to B by one each."""
    c = Circuit(n + 2)
    a = list(range(n))
    p, r = n, n + 1
    cuts = []
    mixer(c, a + [p] if triangle else a)
    if triangle:                                   # p: A, then C; r: C, then B
        cuts.append((p, len(c.gates)))
        c.add(H, r)
        c.add(CX, r, p)
        c.add(S, p)
        c.add(H, p)
        cuts.append((r, len(c.gates)))
    else:                                          # p: C, then D with r
        c.add(H, p)
        c.add(T, p)
        c.add(H, p)
        cuts.append((p, len(c.gates)))
        c.add(CX, p, r)
        c.add(H, r)
    cuts += [(q, len(c.gates)) for q in a]
    mixer(c, a + [r] if triangle else a)
    return Workload("fat", c, cuts, ([0, p, 1, r] + a[2:])[:marginal_bits], [[0, p], [1, r], [0, 1]], 256, 3)


def ring4():
    """Fragments A, B, C, D joined in a ring by two cuts each, three marginal qubits
    in each: two intermediate tensors of 2^6 outcomes x 4^4 cut digits."""
    ab, bc, cd, ad, own = [0, 1], [2, 3], [4, 5], [6, 7], {"A": [8, 9, 10], "B": [11], "C": [12]}
    c = Circuit(13)
    cuts = []
    for start, end, extra in ((ab + ad, [], own["A"]), (bc, ab, own["B"]), (cd, bc, own["C"]), ([], cd + ad, [])):
        cuts += [(q, len(c.gates)) for q in end]
        mixer(c, start + end + extra)
    c.add(T, 4)
    return Workload("ring4", c, cuts, [8, 9, 10, 0, 1, 11, 2, 3, 12, 4, 5, 6], [[0, 8], [3, 5, 6]], 256, 3)


CASES = {
    "pair2": lambda: [fat_edge(2, 3)],
    "pair3_empty": lambda: [fat_edge(3, 0)],
    "pair4": lambda: [fat_edge(4, 4)],
    "pair5_empty": lambda: [fat_edge(5, 0)],
    "pair6": lambda: [fat_edge(6, 2)],
    "pair6_wide": lambda: [fat_edge(6, 8)],
    "triangle2": lambda: [fat_edge(2, 4, True)],
    "triangle4": lambda: [fat_edge(4, 1, True)],
    "triangle5": lambda: [fat_edge(5, 3, True)],
    "ring4": lambda: [ring4()],
    "several": lambda: [fat_edge(2, 4, True), fat_edge(5, 2), fat_edge(3, 3, True), fat_edge(4, 0)],
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("mode", [ccs.CCS_EXACT, ccs.CCS_SAMPLED], ids=["exact", "sampled"])
def test_fat_edges(name, mode):
    ws = CASES[name]()
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, ws)
    for pi in range(len(ws)):
        nf, k = ccs.ccs_plan_counts(ctx, plan, pi)
        assert max(ccs.ccs_fragment_info_get(ctx, plan, pi, f)["n_slots"] for f in range(nf)) < k, "a star"
    res = ccs.ccs_eval_variants(ctx, plan, mode=mode, shots=300)
    m, z = ccs.ccs_recombine(ctx, plan, res)
    half = 4 ** max(len(w.cuts) for w in ws) // 2
    lo, hi = (ccs.ccs_recombine(ctx, plan, res, k_range=r) for r in ((0, half), (half, 0)))
    assert np.abs(m - lo[0] - hi[0]).max() < 2e-6
    assert np.abs(z - lo[1] - hi[1]).max() < 2e-6
    mg, zg = ccs.ccs_recombine(ctx, plan, res, use_graph=True)
    assert np.array_equal(mg, m) and np.array_equal(zg, z)
    if mode == ccs.CCS_EXACT:
        exact = [brute_force(w.circuit, w.marginal, w.zstrings) for w in ws]
        assert np.abs(m - np.concatenate([e[0] for e in exact])).max() < 1e-5
        assert np.abs(z - np.concatenate([e[1] for e in exact])).max() < 1e-5


def test_without_room_for_the_intermediate_tensors(monkeypatch):
    """The request for them is refused by the caller's allocator: the problems are
    then summed directly, as they are over partial ranges."""
    ws = [ring4()]
    asked, refuse = [], []
    real = ccs._TorchAllocator._alloc

    def alloc(self, nbytes, stream, user):
        asked.append(nbytes)
        return None if len(asked) - 1 in refuse else real(self, nbytes, stream, user)
    monkeypatch.setattr(ccs._TorchAllocator, "_alloc", alloc)

    def run():
        ctx = ccs.ccs_create(0)
        plan = ccs.ccs_build_fragments(ctx, ws)
        asked.clear()
        res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_EXACT)
        out = [ccs.ccs_recombine(ctx, plan, res, use_graph=g) for g in (False, True)]
        half = 4 ** max(len(w.cuts) for w in ws) // 2
        parts = [ccs.ccs_recombine(ctx, plan, res, k_range=r) for r in ((0, half), (half, 0))]
        return out, parts[0][0] + parts[1][0]
    out, direct = run()
    refuse.append(asked.index(2 * 4 ** 4 * 2 ** 6 * 8))
    for m, z in run()[0]:
        assert np.abs(m - direct).max() < 2e-6 and np.abs(m - out[0][0]).max() < 2e-6
        assert np.abs(z - out[0][1]).max() < 2e-6
    assert len(asked) > refuse[0]
