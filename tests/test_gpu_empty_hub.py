"""Hubs that measure nothing, beside hubs of twelve to sixteen measured bits (needs a GPU).

A Clifford hub has no measured bit when it has neither a marginal qubit nor a
quantum output: a fragment that is only fed by a cut, with the marginal on the
leaf, or a cut-free circuit with an empty marginal.  All its shots fall on its
one outcome, so such a plan's shot counts, marginals and corrected models must
be the oracle's, also where a wider hub of the same plan decides the width of
the shot counters.  The wider hub's own results are those of a plan of its own
(any counter width gives the same counts, bit for bit).  Bar: 1e-5, the parity
bar of the marginals.
"""
import numpy as np
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import CX, Circuit, H, Region, S, T, Workload, brickwork_star
from oracle.cutting import recombine
from oracle.mlcorrect import ml_correct
from oracle.pipeline import evaluate

pytestmark = pytest.mark.gpu
SEED = (0xE117, 0x0B)


def fed_hub():
    """Qubits 2, 3 carry a T gate and the marginal; qubit 2 then joins the Clifford qubits 0, 1."""
    c = Circuit(4)
    c.add(H, 2)
    c.add(T, 2)
    c.add(H, 2)
    c.add(CX, 2, 3)
    cut = (2, len(c.gates))
    c.add(CX, 2, 0)
    c.add(S, 0)
    c.add(CX, 0, 1)
    return Workload("fed", c, [cut], [3], [], 0, 1)


def cut_free():
    c = Circuit(3)
    c.add(H, 0)
    c.add(CX, 0, 1)
    return Workload("free", c, [], [], [], 0, 1)


def wide(bits):
    """A hub of `bits` measured bits (two of them quantum outputs)."""
    regs = [Region([q], b, 2, 5, [q, b], 1) for q, b in ((0, 1), (6, 7))]
    c, cuts = brickwork_star(24, 10, regs, 5)
    hub = [q for q in range(24) if q not in (0, 6)]
    return Workload("wide", c, cuts, [0, 6] + hub[1:bits - 1], [], 0, 5, regs)


@pytest.mark.parametrize("bits,shots", [(12, 4096), (13, 65535), (16, 1001), (12, 40000)])
@pytest.mark.parametrize("keep", [True, False], ids=["kept", "fast"])
def test_hub_without_measured_bits(bits, shots, keep):
    ws = [wide(bits), fed_hub(), cut_free()]
    ctx = ccs.ccs_create(0)
    kw = dict(mode=ccs.CCS_SAMPLED, shots=shots, seed_lo=SEED[0], seed_hi=SEED[1], keep_tableaus=keep)
    plan = ccs.ccs_build_fragments(ctx, ws)
    # the hub is the first fragment on every cut
    infos = [ccs.ccs_fragment_info_get(ctx, plan, pi, f) for pi, f in ((0, 1), (1, 0), (2, 0))]
    assert [i["n_meas"] for i in infos] == [bits, 0, 0] and all(i["clifford"] for i in infos)
    assert [i["n_slots"] for i in infos] == [ccs.ccs_plan_counts(ctx, plan, pi)[1] for pi in range(3)]
    res = ccs.ccs_eval_variants(ctx, plan, **kw)
    got, _ = ccs.ccs_recombine(ctx, plan, res)
    if keep:
        for pi in (1, 2):
            for v in range(infos[pi]["n_variants"]):
                assert ccs.ccs_get_counts(ctx, res, pi, 0, v).tolist() == [shots]

    alone = ccs.ccs_build_fragments(ctx, ws[:1])
    res_a = ccs.ccs_eval_variants(ctx, alone, **kw)
    want, _ = ccs.ccs_recombine(ctx, alone, res_a)
    assert np.array_equal(got[:want.size], want)

    orcs = [evaluate(w.circuit, w.cuts, w.marginal, (), mode="sampled", shots=shots, seed_lo=SEED[0],
                     seed_hi=SEED[1], circuit_id=pi) for pi, w in ((1, ws[1]), (2, ws[2]))]
    raw = np.concatenate([o.marginal for o in orcs])
    assert np.abs(got[want.size:] - raw).max() < 1e-5
    ccs.ccs_ml_correct(ctx, plan, res)
    got_ml, _ = ccs.ccs_recombine(ctx, plan, res)
    for pi, w, o in ((1, ws[1], orcs[0]), (2, ws[2], orcs[1])):
        models = [ml_correct(f, t)[0] if f.clifford else t for f, t in zip(o.fragments, o.tensors)]
        off = want.size + (0 if pi == 1 else 2)
        m = recombine(o.fragments, models, o.meta["k"], len(w.marginal))
        assert np.abs(got_ml[off:off + m.size] - m).max() < 1e-5
