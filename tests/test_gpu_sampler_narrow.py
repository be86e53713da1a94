"""The hub samplers' counter widths at their edges (needs a GPU).

The default choice takes 4-bit counters for sparse histograms, with the variants
they cannot hold redone by byte counters, 32-bit counters for narrow hubs, and
byte or 16-bit counters otherwise.  Every choice must give the same shot counts,
operands and marginals, bit for bit, also where single outcomes collect many
shots: shallow circuits whose spaces are far from full rank, shots around four
per outcome, partial generator calls, three to twelve marginal bits, none to
four quantum outputs, hubs of different widths in one plan.
"""
import numpy as np
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import CX, Circuit, H, Region, Workload, brickwork_star

pytestmark = pytest.mark.gpu
SEED = (0x1234ABCD, 0x55AA)


def star(n_regions, m_hub, depth=10, seed=1, n=24):
    spots = [(0, 1), (6, 7), (12, 13), (18, 19)][:n_regions]
    regs = [Region([q], b, 2, min(depth - 2, 5), [q, b], 1) for q, b in spots]
    c, cuts = brickwork_star(n, depth, regs, seed)
    hub = [q for q in range(n) if q not in [r.full[0] for r in regs]]
    marg = [r.full[0] for r in regs] + hub[1:1 + m_hub]
    return Workload("star", c, cuts, marg, [], 0, seed, regs)


def few_outcomes(m):
    """A cut-free hub with a two-point space: half the shots on each outcome."""
    c = Circuit(m)
    c.add(H, 0)
    for q in range(1, m):
        c.add(CX, 0, q)
    return Workload("ghz", c, [], list(range(m)), [], 0, 1)


CASES = {   # problems, shots
    "r1_m3": (lambda: [star(1, 3)], 61),
    "r2_m6_sparse": (lambda: [star(2, 6)], 1021),
    "r2_m11_mean4": (lambda: [star(2, 11)], 32000),
    "r2_m11_wide": (lambda: [star(2, 11)], 40000),
    "r3_m10": (lambda: [star(3, 10)], 8191),
    "r3_m10_dense": (lambda: [star(3, 10)], 32767),
    "r4_m9": (lambda: [star(4, 9)], 5000),
    "r4_m10": (lambda: [star(4, 10)], 16384),
    "shallow": (lambda: [star(2, 11, depth=6, seed=3), star(2, 9, depth=6, seed=4)], 2048),
    "ghz": (lambda: [few_outcomes(13), star(2, 11)], 20000),
    "mixed": (lambda: [star(1, 12, seed=7), star(3, 8, seed=8), star(2, 3, seed=9)], 16),
}


@pytest.mark.parametrize("name", list(CASES))
def test_counter_widths_agree(name):
    make, shots = CASES[name]
    ws = make()
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, ws)
    kw = dict(mode=ccs.CCS_SAMPLED, shots=shots, seed_lo=SEED[0], seed_hi=SEED[1], keep_tableaus=True)
    ref = ccs.ccs_eval_variants(ctx, plan, hub_sampler=1, **kw)
    results = [ccs.ccs_eval_variants(ctx, plan, **kw), ccs.ccs_eval_variants(ctx, plan, hub_sampler=2, **kw)]
    # the default path without kept tableaus, replayed from a graph
    fast = ccs.ccs_eval_variants(ctx, plan, use_graph=True, **{**kw, "keep_tableaus": False})
    ccs.ccs_eval_variants(ctx, plan, use_graph=True, res=fast, **{**kw, "keep_tableaus": False})
    m_ref, _ = ccs.ccs_recombine(ctx, plan, ref)
    for r in results + [fast]:
        m, _ = ccs.ccs_recombine(ctx, plan, r)
        assert np.array_equal(m, m_ref)
    for pi in range(len(ws)):
        nf, k = ccs.ccs_plan_counts(ctx, plan, pi)
        for f in range(nf):
            info = ccs.ccs_fragment_info_get(ctx, plan, pi, f)
            if not info["clifford"] or info["n_slots"] != k:
                continue
            want = ccs.ccs_get_operand(ctx, ref, pi, f)
            assert all(np.array_equal(ccs.ccs_get_operand(ctx, r, pi, f), want) for r in results + [fast])
            for v in range(0, info["n_variants"], max(1, info["n_variants"] // 40)):
                counts = ccs.ccs_get_counts(ctx, ref, pi, f, v)
                assert int(counts.sum()) == shots
                assert all(np.array_equal(ccs.ccs_get_counts(ctx, r, pi, f, v), counts) for r in results)
