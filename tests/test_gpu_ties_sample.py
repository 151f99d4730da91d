"""TIES thresholds at the edges of the sampling rule and of the warp-wide selects.

The sample takes 8, 32 or up to 128 vectors of a block by the number of blocks in its trim
group (256 or more, 64 or more, fewer), groups of 16 blocks or more get a narrow window; the
selects give each lane a run of 4, 8, 12 or 20 bins.
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
@pytest.mark.parametrize("n_b", [1, 15, 16, 63, 64, 65, 255, 256])
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


def _sampled_vectors(b, n_b, nvec, nvec0):
    """the vectors of block b that the sample reads"""
    want = 8 if n_b >= 256 else (32 if n_b >= 64 else 128)
    n_v = min(max((want * nvec + nvec0 // 2) // nvec0, 1), nvec)
    if n_v == nvec:
        return np.arange(nvec)
    v0 = np.arange(n_v, dtype=np.uint64)
    h = (np.uint64(b) * np.uint64(0x9E3779B1) & np.uint64(0xFFFFFFFF)) ^ ((v0 + 1) * np.uint64(0x85EBCA77) & np.uint64(0xFFFFFFFF))
    h ^= h >> np.uint64(15)
    h = h * np.uint64(0x2C1B3C6D) & np.uint64(0xFFFFFFFF)
    h ^= h >> np.uint64(12)
    per = nvec // n_v
    return (v0 * per + h % np.uint64(per)).astype(np.int64)


@pytest.mark.parametrize("n_b,blk", [(3, 65536), (20, 65536), (70, 4096)])
def test_a_sample_that_sees_only_outliers_falls_back(n_b, blk):
    """Deltas of 0.5 exactly where the sample reads and small ones everywhere else: the window
    lies among the outliers, the threshold among the small deltas, and the two-level select of
    the marked pairs must give the oracle's threshold (with whole binades and with narrow windows,
    and with a partial last block)."""
    import torch

    fam = synth.custom([n_b * blk - 808, 4096], dtype=synth.BF16, block_elems=blk, K=5, active_frac=0.5, name="outliers")
    base, experts = fam.host_arrays()
    bo, bl, bt = fam.block_table()
    f32 = lambda x: (x.astype(np.uint32) << 16).view(np.float32)  # noqa: E731
    rng = np.random.default_rng(8)
    for i in range(fam.K):
        d = (1e-3 * rng.standard_normal(base.size)).astype(np.float32)
        for b in np.nonzero(bt == 0)[0]:
            for v in _sampled_vectors(int(b), n_b, (int(bl[b]) + 7) // 8, blk // 8):
                d[int(bo[b]) + 8 * v:int(bo[b]) + 8 * v + 8] = 0.5
        experts[i] = torch.from_numpy(f32(base) + d).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
    mf, _, _ = upload(fam, base, experts)
    idx = mp.mp_index_blocks(mf, mp.make_op(mp.MP_OP_TIES, lam=1.0, density=0.2))
    tau = mp.mp_index_stats(idx)[3]
    idx.free()
    assert np.array_equal(tau, oracle.ties_thresholds(oracle_family(fam, base, experts), float(np.float32(0.2))))
    assert np.all(tau[:, 0] < 0x3E00)  # bf16 key of 0.125: far below the sampled outliers
