"""Edges of the maximum-likelihood correction's block kernels (needs a GPU).

Blocks of 16, 32 and 64 rows keep their columns in registers; 16-row blocks
share warps, also across fragments of different kinds.  One plan holds hubs of
four, five and six cut slots with one and with a few outcomes (an odd number of
blocks in all), a four-slot fragment inside a tree and a cut-free circuit with
an empty marginal; at few shots some outcomes are never seen (zero blocks).
Bars as for the correction itself: T' within 4 N 2^-24 (N = 2^(d+1)) of the
FP64 oracle relative to max(1, max |T|), marginals within 1e-5.
"""
import numpy as np
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import CX, Circuit, H, Region, Workload, brickwork_star, tree_circuit
from oracle.cutting import recombine
from oracle.mlcorrect import ml_correct
from oracle.pipeline import evaluate

pytestmark = pytest.mark.gpu
SEED = (0xB10C, 0x5EED)


def star(n_regions, marginal, seed, open_end=False):
    spots = [(0, 1), (7, 8), (15, 14)][:n_regions]
    regs = [Region([q], b, 2, 10 if open_end and i == n_regions - 1 else 5 + i, [q, b], 1)
            for i, (q, b) in enumerate(spots)]
    c, cuts = brickwork_star(16, 10, regs, seed)
    return Workload("star", c, cuts, marginal, [], 0, seed, regs)


def tree():
    c, cuts = tree_circuit([0, 0, 0, 0, 1], 12, 1, seed=6)
    return Workload("tree", c, cuts, [1, 5, 16], [], 0, 6)


def cut_free():
    c = Circuit(3)
    c.add(H, 0)
    c.add(CX, 0, 1)
    return Workload("free", c, [], [], [], 0, 1)


@pytest.mark.parametrize("shots", [8, 200])
def test_blocks_match_oracle(shots):
    ws = [cut_free(), star(2, [0, 7], 5), star(2, [0, 7, 3, 11], 6), tree(), star(3, [0, 7, 15], 7),
          star(3, [0, 7, 15, 4, 11], 8), star(3, [7, 15], 9, open_end=True), star(2, [3], 10)]
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, ws)
    res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=shots, seed_lo=SEED[0], seed_hi=SEED[1])
    ccs.ccs_ml_correct(ctx, plan, res)
    m, _ = ccs.ccs_recombine(ctx, plan, res)
    off, sizes = 0, set()
    for pi, w in enumerate(ws):
        orc = evaluate(w.circuit, w.cuts, w.marginal, (), mode="sampled", shots=shots, seed_lo=SEED[0],
                       seed_hi=SEED[1], circuit_id=pi)
        want = [ml_correct(f, T)[0] if f.clifford else T for f, T in zip(orc.fragments, orc.tensors)]
        for fi, (f, Tw) in enumerate(zip(orc.fragments, want)):
            got = ccs.ccs_get_tensor(ctx, res, pi, fi).astype(np.float64)
            bar = 4.0 * (2 << len(f.slots)) * 2.0 ** -24 * max(1.0, np.abs(Tw).max())
            if f.clifford:
                sizes.add(len(f.slots))
            assert np.abs(got - Tw).max() < bar, (pi, fi, len(f.slots))
        want_m = recombine(orc.fragments, want, orc.meta["k"], len(w.marginal))
        assert np.abs(m[off:off + want_m.size] - want_m).max() < 1e-5, pi
        off += want_m.size
    assert {0, 4, 5, 6} <= sizes
