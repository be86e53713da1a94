"""A result evaluated again with another number of shots and recombined from its
CUDA graph (needs a GPU): the replay must equal direct launches bit for bit,
whichever of the shot counts the graph was captured with, over the leaf-by-leaf
contraction, the streaming GEMM and the tensor-core GEMM, with 16-bit count
sums (up to 32767 shots) and FP32 operands, and after a correction."""
import numpy as np
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import Region, Workload, brickwork_star, config2

pytestmark = pytest.mark.gpu


def wide_star():
    regs = [Region([0, 1], 2, 2, 6, [0, 1], 1), Region([11, 12], 13, 3, 7, [11, 12], 1),
            Region([22, 23], 21, 2, 5, [22, 23], 1)]
    c, cuts = brickwork_star(24, 9, regs, 5)
    return Workload("star3", c, cuts, [0, 1, 11, 22] + [3, 4, 5, 6, 7, 8, 9, 15], [], 300, 5, regs)


@pytest.mark.parametrize("make", [config2, wide_star])
@pytest.mark.parametrize("precision", [ccs.CCS_FP32, ccs.CCS_BF16])
def test_replay_after_other_shots(make, precision):
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, [make()])
    res = None
    for shots, correct in ((1000, False), (3000, False), (40000, False), (3000, False), (3000, True), (1000, False)):
        res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=shots, res=res, use_graph=True)
        if correct:
            ccs.ccs_ml_correct(ctx, plan, res)
        want, zw = ccs.ccs_recombine(ctx, plan, res, precision=precision)
        for _ in range(2):
            got, z = ccs.ccs_recombine(ctx, plan, res, precision=precision, use_graph=True)
            assert np.array_equal(got, want) and np.array_equal(z, zw), (shots, correct)
