"""TIES thresholds at the edges of the sampling rule and of the warp-wide selects.

The sample takes 8, 32 or up to 128 vectors of a block by the number of blocks in its trim
group (64 or more, 16 or more, fewer); the selects give each lane a run of 4, 8 or 12 bins.
Group sizes on both sides of each line, one-vector tensors, and ranks from the largest key
(k = 1) to the smallest (k = numel) must give the oracle's thresholds.
"""
import numpy as np
import pytest

import oracle
from conftest import oracle_family
from test_gpu_parity import upload

pytestmark = pytest.mark.gpu

import paper_2605_29489_gb300 as mp  # noqa: E402
from paper_2605_29489_gb300 import synth  # noqa: E402

E = 1024


@pytest.mark.parametrize("dtype", [synth.BF16, synth.F32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("n_b", [1, 15, 16, 63, 64, 65])
def test_thresholds_at_the_edges_of_the_sampling_rule(n_b, dtype):
    fam = synth.custom([n_b * E - 5, 3, 8, n_b * E // 2 + 1], dtype=dtype, block_elems=E, K=5, active_frac=0.6,
                       name="sample-edges")
    base, experts = fam.host_arrays()
    mf, _, _ = upload(fam, base, experts)
    for scope in (0, 1):
        for density in (1.0 / (n_b * E - 5), 0.2, 1.0):
            idx = mp.mp_index_blocks(mf, mp.make_op(mp.MP_OP_TIES, lam=1.0, density=density, trim_scope=scope))
            tau = mp.mp_index_stats(idx)[3]
            want = oracle.ties_thresholds(oracle_family(fam, base, experts, scope), float(np.float32(density)))
            assert np.array_equal(tau, want), (scope, density)
            idx.free()
