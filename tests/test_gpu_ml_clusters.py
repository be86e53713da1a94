"""Correction of blocks whose eigenvalues lie in tight clusters (needs a GPU).

With very many shots a fragment's Choi blocks are close to those of an exact
Clifford channel: one eigenvalue of order one and all others within the small
shot noise (every wire of the fragment cut), one value and noise (its outputs
replaced by fresh maximally mixed qubits), or two clusters.  Inside a cluster the eigenvectors turn by large angles however
small the off-diagonals are, so an eigensolver must not stop before these have
vanished to rounding.

Bar: ||T' - T'_ref||_2 <= N 2^-24 ||T'_ref||_2 against the FP64 oracle on the
same shot counts, N = 2^(d+1) the real dimension of a complex block: the backward
error bound N eps of a dense FP32 eigendecomposition, T and J having the same
Frobenius norm up to a factor.
"""
import numpy as np
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import CX, CZ, H, S, T, Circuit, Workload
from oracle.cutting import fold, fragment_circuit
from oracle.mlcorrect import ml_correct

pytestmark = pytest.mark.gpu


def channel(n, nin, mixed=0):
    """A Clifford hub on n wires, all cut at its end and the first nin at its start
    (T gates beyond the cuts); the first `mixed` leave it as halves of fresh
    entangled pairs."""
    c = Circuit(n + 2 * mixed)
    cuts = []
    for q in range(nin):
        c.add(H, q)
        c.add(T, q)
        c.add(H, q)
        cuts.append((q, len(c.gates)))
    for layer in range(4):
        for q in range(n):
            c.add(H, q)
            c.add(S, (q + layer) % n)
            c.add(CX if (q + layer) % 2 else CZ, q, (q + 1) % n)
    for i in range(mixed):
        a, b = n + 2 * i, n + 2 * i + 1
        c.add(H, a)
        c.add(CX, a, b)
        for x, y in ((i, a), (a, i), (i, a)):
            c.add(CX, x, y)
    for q in range(n):
        cuts.append((q, len(c.gates)))
        c.add(H, q)
        c.add(T, q)
        c.add(H, q)
    return Workload("channel", c, cuts, list(range(n)), [], 0, 1)


CASES = [   # wires, of them cut at the start, mixed, shots, seed: blocks of 16, 32 and 64 rows
    (4, 0, 0, 2 ** 31, 1), (4, 0, 0, 2 ** 31, 2), (4, 0, 0, 2 ** 32 - 1, 3), (4, 0, 0, 2 ** 30, 4),
    (5, 0, 0, 2 ** 31, 5), (5, 0, 0, 2 ** 32 - 1, 6), (6, 0, 0, 2 ** 31, 7),
    (2, 2, 2, 2 ** 22, 8), (3, 3, 3, 2 ** 22, 9), (3, 3, 1, 2 ** 24, 10),
]


@pytest.mark.parametrize("n,nin,mixed,shots,seed", CASES)
def test_clustered_blocks(n, nin, mixed, shots, seed):
    w = channel(n, nin, mixed)
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, [w])
    frags, cuts = fragment_circuit(w.circuit, w.cuts, w.marginal)
    hub = [i for i, f in enumerate(frags) if len(f.slots) == len(cuts)][0]
    f = frags[hub]
    assert f.clifford and len(f.slots) == n + nin
    res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=shots, seed_lo=seed, seed_hi=9,
                                keep_tableaus=True)
    raw = fold(f, [ccs.ccs_get_counts(ctx, res, 0, hub, v) / float(shots) for v in range(f.n_variants)])
    want, _ = ml_correct(f, raw)
    ccs.ccs_ml_correct(ctx, plan, res)
    err = np.linalg.norm(ccs.ccs_get_tensor(ctx, res, 0, hub).astype(np.float64) - want)
    bar = (2 << len(f.slots)) * 2.0 ** -24 * np.linalg.norm(want)
    assert err < bar, err / bar
