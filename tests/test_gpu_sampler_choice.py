"""Which hub sampler a result uses (needs a GPU): a sparse plan of wide hubs
starts with 4-bit counters; a caller's own choice, or more shots than those
hold, then gets the CTA shape of the counters it runs with.

The operands read out of 32-bit counters (more than 65535 shots, and narrow
hubs) are compared with sums of the dense counts: whole numbers of at most
2^26, rounded to FP32 once and scaled by 1 / shots rounded to FP32, so within
three half-ulps."""
import itertools

import numpy as np
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import Region, Workload, brickwork_star

pytestmark = pytest.mark.gpu


def star(m_hub, n=24, regions=2, open_ends=0):
    """Two cuts per region (one where the last `open_ends` run to the circuit's end)."""
    spots = ((6, 7), (0, 1), (12, 13), (18, 19))[:regions]
    regs = [Region([q], b, 2, 10 if i >= regions - open_ends else 5, [q, b], 1) for i, (q, b) in enumerate(spots)]
    c, cuts = brickwork_star(n, 10, regs, 5)
    full = [q for q, _ in spots]
    hub = [q for q in range(n) if q not in full and q not in [b for _, b in spots[regions - open_ends:]]]
    return Workload("star", c, cuts, full + hub[1:1 + m_hub], [], 0, 5, regs)


@pytest.fixture(scope="module")
def sparse():
    """A plan of one hub of 13 measured bits and its result at 4096 shots."""
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, [star(11)])
    return ctx, plan


def evaluate(sparse, **kw):
    ctx, plan = sparse
    res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=4096)
    assert ccs.ccs_get_tuning(ctx, res)[3] == -128
    if kw:
        ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, res=res, **kw)
    return ccs.ccs_get_tuning(ctx, res)[3]


def test_forced_16_bit_counters_take_512_threads(sparse):
    assert evaluate(sparse, shots=4096, hub_sampler=1) == 512


@pytest.mark.parametrize("shots,want", [(32767, -128), (32768, -256), (65535, -256), (65536, 256)])
def test_reported_counters_are_those_of_the_last_evaluation(sparse, shots, want):
    """13 measured bits: 4-bit counters up to four shots per outcome and 32767
    shots, byte counters up to 65535."""
    assert evaluate(sparse, shots=shots) == want


def test_tuned_shapes_are_kept_per_kind_of_hub():
    """Two plans of one shape bucket, the second's hub too narrow for byte and
    4-bit counters: it is tuned for itself, and reports neither."""
    ctx = ccs.ccs_create(0)
    launches = []
    for m in (11, 1, 1):
        plan = ccs.ccs_build_fragments(ctx, [star(m)])
        before = ccs.ccs_launch_count()
        res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=4096, autotune=True)
        launches.append(ccs.ccs_launch_count() - before)
    assert ccs.ccs_get_tuning(ctx, res)[3] > 0
    # the third takes the second's shape from the cache: one evaluation's launches
    assert launches[1] > 4 * launches[2] > 0


def test_narrow_hubs_keep_128_threads():
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, [star(8)])
    res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=4096)
    assert ccs.ccs_get_tuning(ctx, res)[3] == 128
    ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=4096, res=res, hub_sampler=1)
    assert ccs.ccs_get_tuning(ctx, res)[3] == 128


@pytest.mark.parametrize("m,regions,open_ends,shots", [
    (0, 1, 0, 40000), (1, 1, 1, 70001), (3, 2, 0, 32768), (8, 2, 1, 65535), (12, 3, 0, 70000), (4, 2, 2, 100000),
    (11, 4, 1, 66000), (5, 2, 0, 1 << 26), (0, 2, 0, 1000)])
def test_operands_of_32_bit_counters(m, regions, open_ends, shots):
    ctx = ccs.ccs_create(0)
    w = star(m, regions=regions, open_ends=open_ends)
    plan = ccs.ccs_build_fragments(ctx, [w])
    nf, k = ccs.ccs_plan_counts(ctx, plan, 0)
    res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=shots, keep_tableaus=True)
    from oracle.cutting import fragment_circuit
    frags, _ = fragment_circuit(w.circuit, w.cuts, w.marginal)
    hub = [i for i, f in enumerate(frags) if len(f.slots) == k and f.clifford][0]
    f = frags[hub]
    qi, qo, mh = len(f.qin), len(f.qout), len(f.marg)
    place = {c: j for j, c in enumerate(f.slots)}
    got = ccs.ccs_get_operand(ctx, res, 0, hub).astype(np.float64)
    bits = np.arange(1 << qo)
    for v in range(0, f.n_variants, max(1, f.n_variants // 60)):
        counts = ccs.ccs_get_counts(ctx, res, 0, hub, v).astype(np.int64).reshape(1 << qo, 1 << mh)
        assert counts.sum() == shots
        preps, bases = f.variant_digits(v)
        # each output: the Pauli of its basis (X, Y), or I and Z
        for paulis in itertools.product(*[((0, 3) if b == 2 else (b + 1,)) for b in bases]):
            mask = sum(1 << j for j, p in enumerate(paulis) if p)
            sign = 1 - 2 * (np.array([bin(int(x) & mask).count("1") for x in bits]) & 1)
            d = sum(s << (2 * place[c]) for s, (c, _) in zip(preps, f.qin))
            d += sum(p << (2 * place[c]) for p, (c, _) in zip(paulis, f.qout))
            want = (sign[:, None] * counts).sum(0) / shots
            assert np.all(np.abs(got[:, d] - want) <= 3 * 2.0 ** -24 * np.abs(want) + 1e-45)
    assert qi <= 4 and qo <= 4
