"""TIES after masking from the units' histograms.

Where blocks are large the catalog keeps, for each (expert, block), the counts of 384 keys around
the predicted threshold and of the binades outside them; a plan's thresholds come from the sums
over the blocks it selects.  Catalogs, plans and merges must be the oracle's whether a threshold
lies inside its window, far below it (small budgets leave out most of the large deltas) or among
the zeros, on both sides of the line on the block size, and when the sample misleads.
"""
import numpy as np
import pytest

from test_gpu_parity import run_case
from test_gpu_ties_sample import _sampled_vectors

pytestmark = pytest.mark.gpu

from paper_2605_29489_gb300 import synth  # noqa: E402

LINE = 2048  # elements of a block on average from which the larger histograms are kept
FRACS = [0.02, 0.1, 0.2, 0.3, 0.5, 0.8, 1.0]


@pytest.mark.parametrize("dtype", [synth.BF16, synth.F32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("K", [1, 2, 3, 6])
@pytest.mark.parametrize("block", [LINE - 8, LINE, 40000], ids=["below", "at", "above"])
def test_thresholds_of_plans(block, K, dtype):
    n = block
    fam = synth.custom([40 * n, 9 * n], dtype=dtype, block_elems=n, K=K, active_frac=0.6, per_expert_active=K == 6,
                       name=f"units-{block}-{K}", log_sigma=1.5)
    base, experts = fam.host_arrays()
    run_case(fam, base, experts, ("ties_masked", "ties_masked1"), FRACS)


def test_sample_that_misleads():
    """outliers where the sample reads (the window lies among them), small deltas elsewhere"""
    import torch

    fam = synth.custom([20 * 65536 - 808, 4096], dtype=synth.BF16, block_elems=65536, K=5, active_frac=0.5,
                       name="units-outliers")
    base, experts = fam.host_arrays()
    bo, bl, bt = fam.block_table()
    rng = np.random.default_rng(8)
    for i in range(fam.K):
        d = (1e-3 * rng.standard_normal(base.size)).astype(np.float32)
        for b in np.nonzero(bt == 0)[0]:
            for v in _sampled_vectors(int(b), 20, (int(bl[b]) + 7) // 8, 65536 // 8):
                d[int(bo[b]) + 8 * v:int(bo[b]) + 8 * v + 8] = 0.5
        x = torch.from_numpy((base.astype(np.uint32) << 16).view(np.float32) + d)
        experts[i] = x.to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
    run_case(fam, base, experts, ("ties_masked", "ties_masked1"), [0.1, 0.5, 1.0])
