"""BF16 contractions against bars on each output's own scale (needs a GPU).

Tensor cores: a star's sampled hub operand Q (16-bit count sums times 1 / shots)
and the leaves' FP32 product R are rounded to bf16 and multiplied exactly, so
output o differs from the FP64 product of the rounded operands only by FP32
accumulation: chains of at most 1024 additions, each of 2^-24 (the tensor core
may truncate: 2^-23) of the sum of absolute terms A(o) = 2^-k sum |Q| |R|.  Bar:
3072 2^-24 A(o).  That it would see a wrong layout is asserted: the outputs
shifted by one place, and zeros, are outside of it nearly everywhere.

Trees: every fragment tensor is rounded to bf16 and the rest is FP64, so the
result is the FP64 contraction of the rounded tensors; bar 2^-40 A(o).
"""
import numpy as np
import pytest
import torch

from paper_2303_10788_gb300 import ccs
from workloads import Region, Workload, brickwork_star, tree_circuit
from oracle.cutting import fragment_circuit, recombine

pytestmark = pytest.mark.gpu


def star(hub_bits, leaf_bits, seed=5):
    n = 24
    regs = [Region([0, 1], 2, 2, 6, [0, 1], 1), Region([11, 12], 13, 3, 7, [11, 12], 1),
            Region([22, 23], 21, 2, 5, [22, 23], 1)]
    c, cuts = brickwork_star(n, 9, regs, seed)
    leaf = [0, 11, 22, 1, 12, 23][:leaf_bits]
    hub = [q for q in range(3, 21) if q not in (11, 12)][:hub_bits]
    return Workload("star3", c, cuts, sorted(hub + leaf), [], 300, seed, regs)


@pytest.mark.parametrize("hub_bits,leaf_bits,shots", [(7, 4, 300), (9, 4, 32767), (8, 5, 3000), (11, 5, 16384)])
def test_counts_gemm_on_the_outputs_scale(hub_bits, leaf_bits, shots):
    w = star(hub_bits, leaf_bits)
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, [w])
    res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=shots)
    got, _ = ccs.ccs_recombine(ctx, plan, res, precision=ccs.CCS_BF16)
    frags, cuts = fragment_circuit(w.circuit, w.cuts, w.marginal)
    k = len(cuts)
    hub = [i for i, f in enumerate(frags) if len(f.slots) == k][0]
    P, o = np.arange(4 ** k), np.arange(1 << len(w.marginal))

    def local(f):                                # a fragment's own outcome of every output
        return sum((((o >> mi) & 1) << j for j, (mi, _) in enumerate(f.marg)), np.zeros_like(o))
    R, n, off = np.ones((4 ** k, 1 << leaf_bits), np.float32), np.zeros_like(o), 0
    for i, f in enumerate(frags):
        if i == hub:
            continue
        x = (np.arange(1 << leaf_bits) >> off) & ((1 << len(f.marg)) - 1)
        pf = sum((((P >> (2 * c)) & 3) << (2 * j) for j, c in enumerate(f.slots)), np.zeros_like(P))
        R *= ccs.ccs_get_operand(ctx, res, 0, i)[x[None, :], pf[:, None]]
        n |= local(f) << off
        off += len(f.marg)
    Q, R = (torch.from_numpy(a).bfloat16().double().numpy() for a in (ccs.ccs_get_operand(ctx, res, 0, hub), R))
    at = (local(frags[hub]), n)
    want = (Q @ R)[at] / 2.0 ** k
    bar = 3072 * 2.0 ** -24 * (np.abs(Q) @ np.abs(R))[at] / 2.0 ** k
    assert np.all(np.abs(got - want) <= bar)
    seen = np.abs(want) > bar                    # (some leaf qubits are certain: zeros beside them)
    assert seen.mean() >= 0.25
    for wrong in (np.zeros_like(want), np.roll(want, 1), np.roll(want, 1 << leaf_bits)):
        assert (np.abs(wrong - want)[seen] > bar[seen]).mean() > 0.9


@pytest.mark.parametrize("parents,marg", [([0, 1, 2], list(range(6))), ([0, 0, 1, 1], list(range(12))),
                                          ([0, 1, 2, 3, 4], [0, 7, 16])])
def test_trees_round_the_tensors_only(parents, marg):
    c, cuts = tree_circuit(parents, 14, 3, seed=1)
    w = Workload("tree", c, cuts, [q % c.n_qubits for q in marg], [], 256, 3)
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, [w])
    res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=300)
    got, _ = ccs.ccs_recombine(ctx, plan, res, precision=ccs.CCS_BF16)
    frags, cc = fragment_circuit(w.circuit, w.cuts, w.marginal)
    ts = [torch.from_numpy(ccs.ccs_get_tensor(ctx, res, 0, i)).bfloat16().double().numpy() for i in range(len(frags))]
    want = recombine(frags, ts, len(cc), len(w.marginal))
    absum = recombine(frags, [np.abs(t) for t in ts], len(cc), len(w.marginal))
    assert np.all(np.abs(got - want) <= 2.0 ** -40 * absum)
