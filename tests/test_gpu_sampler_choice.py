"""Which hub sampler a result uses (needs a GPU): a sparse plan of wide hubs
starts with 4-bit counters; a caller's own choice, or more shots than those
hold, then gets the CTA shape of the counters it runs with."""
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import Region, Workload, brickwork_star

pytestmark = pytest.mark.gpu


def star(m_hub, n=24):
    regs = [Region([q], b, 2, 5, [q, b], 1) for q, b in ((0, 1), (6, 7))]
    c, cuts = brickwork_star(n, 10, regs, 5)
    hub = [q for q in range(n) if q not in (0, 6)]
    return Workload("star", c, cuts, [0, 6] + hub[1:1 + m_hub], [], 0, 5, regs)


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


def test_narrow_hubs_keep_128_threads():
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, [star(8)])
    res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=4096)
    assert ccs.ccs_get_tuning(ctx, res)[3] == 128
    ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=4096, res=res, hub_sampler=1)
    assert ccs.ccs_get_tuning(ctx, res)[3] == 128
