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


def test_little_memory_takes_the_smaller_histograms():
    """1.28 million units: 3.3 GB with the larger histograms, 1.3 GB with the smaller ones; with 2.4 GB
    free the catalog takes the latter, and the thresholds, the plan and the output are the same"""
    import torch

    import paper_2605_29489_gb300 as mp

    n, K = 2048 * 40000, 32
    g = torch.Generator(device="cuda").manual_seed(5)
    base = torch.randn(n, generator=g, device="cuda").mul_(0.02).to(torch.bfloat16)
    expert = (base.float() + 1e-3 * torch.randn(n, generator=g, device="cuda")).to(torch.bfloat16)
    fam = mp.family([(0, n // 2), (n // 2, n // 2)], base, [expert] * K, 2048, mp.MP_BF16, 0)
    op = mp.make_op(mp.MP_OP_TIES_MASKED, lam=1.0, density=0.2)

    def run():
        out = torch.zeros_like(base)
        with mp.mp_index_blocks(fam, op) as idx:
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            tau = mp.mp_index_stats(idx)[3]
            with mp.mp_plan(idx, op, mp.mp_budget_from_fraction(fam, 0.3)) as plan:
                with mp.mp_merge(fam, idx, plan, out) as man:
                    digest = mp.mp_manifest_info(man, K)["digest"]
        return tau, digest, out, free

    tau, digest, out, _ = run()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (2400 << 20), dtype=torch.uint8, device="cuda")
    tau2, digest2, out2, free = run()
    assert free > 512 << 20  # the larger histograms would not have fitted
    del hold
    torch.cuda.empty_cache()  # not kept by torch's allocator: other tests look at what is free
    assert np.array_equal(tau, tau2) and digest == digest2
    assert torch.equal(out.view(torch.int16), out2.view(torch.int16))
