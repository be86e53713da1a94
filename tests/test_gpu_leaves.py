"""Statevector leaves and the leaf-by-leaf contraction at their edges (needs a GPU).

Leaves of 2 to 10 wires: four lanes per group of amplitudes up to 8 wires, one
from 9 on, several widths in one plan.  Z-strings on both sides of the line at
which a warp takes each instead of a CTA; marginals that give one, a few and
many slices per hub.  Everything is compared with the uncut statevector; the
bar is the parity bar, 1e-5.  A leaf here is at most 90 fused ops, each at most
eight roundings of 2^-24 of the norm, adding like sqrt(90): 4.5e-6.
"""
import numpy as np
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import small_star
from oracle.pipeline import brute_force

pytestmark = pytest.mark.gpu


def star(width, n_marg=3, n_z=8, seed=1):
    full = tuple(range(width - 1))
    n = max(width + 4, n_marg)
    marg = [int(q) for q in np.random.default_rng(seed).permutation(n)[:n_marg]]
    return small_star(n=n, depth=9, region_full=full, boundary=width - 1, window=(2, 6), n_t=2, marginal=marg,
                      seed=seed, n_z=n_z)


CASES = {f"wires{w}": [(w,)] for w in range(2, 11)}
CASES["mixed"] = [(2,), (8,), (10,), (5,)]
CASES["mixed_small"] = [(8,), (3,), (7,)]
CASES["strings150"] = [(6, 3, 50, s) for s in range(3)]
CASES["strings180"] = [(6, 3, 60, s) for s in range(3)]
CASES["marginal0"] = [(5, 0)]
CASES["marginal10"] = [(5, 10)]
CASES["marginals"] = [(4, 8, 1, s) for s in range(12)] + [(6, 1)]


@pytest.mark.parametrize("name", list(CASES))
def test_leaves_equal_uncut_statevector(name):
    ws = [star(*a) for a in CASES[name]]
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, ws)
    for pi, (w, a) in enumerate(zip(ws, CASES[name])):
        nf, _ = ccs.ccs_plan_counts(ctx, plan, pi)
        infos = [ccs.ccs_fragment_info_get(ctx, plan, pi, f) for f in range(nf)]
        assert a[0] in [i["n_wires"] for i in infos if not i["clifford"]]
    res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_EXACT)
    exact = [brute_force(w.circuit, w.marginal, w.zstrings) for w in ws]
    for graph in (False, True):
        m, z = ccs.ccs_recombine(ctx, plan, res, use_graph=graph)
        assert np.abs(m - np.concatenate([e[0] for e in exact])).max() < 1e-5
        assert np.abs(z - np.concatenate([e[1] for e in exact])).max() < 1e-5
