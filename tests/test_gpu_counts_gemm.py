"""The BF16 tensor-core contraction reading a sampled hub's 16-bit count sums (needs a GPU).

Stars with six cuts: K = 4096 cut indices, 16 or 32 leaf outputs, one to sixteen
tiles of 128 hub outputs.  The tensor-core path (counts converted inside the
GEMM) is compared with the same contraction on CUDA cores: both round the same
operands to bf16 and multiply exactly, so they differ by FP32 accumulation only
-- at most 256 products of absolute sum <= 1 per accumulator, 256 * 2^-24 of it
(1.6e-5); K terms scaled by 2^-6 with |Q| <= 1, |R| <= 2^6 keep the sum of
absolute terms of an output within K.  Measured against the outputs' own scale
the bar is 2e-5, plus the uncorrected FP32 sums of the CUDA-core tile.  A second
evaluation with more shots than 16 bits hold takes the FP32 operand's path.
"""
import numpy as np
import pytest

from paper_2303_10788_gb300 import ccs
from workloads import Region, Workload, brickwork_star

pytestmark = pytest.mark.gpu


def star(hub_bits, leaf_bits, seed=5):
    n = 24
    regs = [Region([0, 1], 2, 2, 6, [0, 1], 1), Region([11, 12], 13, 3, 7, [11, 12], 1),
            Region([22, 23], 21, 2, 5, [22, 23], 1)]
    c, cuts = brickwork_star(n, 9, regs, seed)
    leaf = [0, 11, 22, 1, 12, 23][:leaf_bits]
    hub = [q for q in range(3, 21) if q not in (11, 12)][:hub_bits]
    return Workload("star3", c, cuts, sorted(hub + leaf), [], 300, seed, regs)


@pytest.mark.parametrize("hub_bits,leaf_bits", [(7, 4), (8, 5), (9, 4), (11, 5), (11, 4)])
@pytest.mark.parametrize("shots", [300, 32767, 40000])
def test_counts_gemm_equals_cuda_cores(hub_bits, leaf_bits, shots):
    ws = [star(hub_bits, leaf_bits)]
    ctx = ccs.ccs_create(0)
    plan = ccs.ccs_build_fragments(ctx, ws)
    res = ccs.ccs_eval_variants(ctx, plan, mode=ccs.CCS_SAMPLED, shots=shots)
    exact, _ = ccs.ccs_recombine(ctx, plan, res)
    want, _ = ccs.ccs_recombine(ctx, plan, res, precision=ccs.CCS_BF16, tensor_cores=False)
    for graph in (False, True):
        got, _ = ccs.ccs_recombine(ctx, plan, res, precision=ccs.CCS_BF16, use_graph=graph)
        assert np.abs(got - want).max() < 2e-5
        assert np.abs(got - exact).max() < 1e-2
