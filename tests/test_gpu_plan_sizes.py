"""The planner at the edges of its launch sizes, from imported catalogs, against the oracle.

Unit counts on both sides of one CTA, of each cluster size and of the line between the cluster and
the cooperative launch (2^17 units); catalogs whose scores share digits (sort passes that move
nothing), tie, or are zero; tails of unequal costs longer than one chunk, where the greedy takes
whole chunks, parts of them, and skips; budgets from nothing to everything; a kept order reused.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

import paper_2605_29489_gb300 as mp  # noqa: E402


def _check(numels, E, K, norms, budgets, zero_frac=0.0, missing=0.0, score_mode=0, seed=0):
    offs, o = [], 0
    for n in numels:
        offs.append(o)
        o += (n + 7) // 8 * 8
    base = torch.zeros(o, dtype=torch.bfloat16, device="cuda")
    other = torch.zeros_like(base)  # never read: the catalog is imported
    fam = mp.family(list(zip(offs, numels)), base, [other] * K, E, mp.MP_BF16, 0)
    bl = np.concatenate([np.minimum(E, n - np.arange(0, n, E)) for n in numels]).astype(np.uint32)
    bt = np.concatenate([np.full((n + E - 1) // E, t) for t, n in enumerate(numels)]).astype(np.uint32)
    rng = np.random.default_rng(seed)
    nb = bl.size
    norm = norms(rng, (K, nb)).astype(np.float32)
    nnz = np.minimum(bl, 1 + rng.integers(0, E, (K, nb))).astype(np.uint32)
    nnz[rng.random((K, nb)) < zero_frac] = 0
    if missing:
        nnz[rng.random((K, nb)) < missing] = mp.MP_NNZ_MISSING
    alpha = [0.3 + 0.1 * (i % 3) for i in range(K)]
    gop = mp.make_op(mp.MP_OP_TA, alpha=alpha, score_mode=score_mode)
    oop = oracle.Op(oracle.TA, K, alpha=alpha, score_mode=score_mode)
    idx = mp.mp_index_import(fam, gop, norm, norm, nnz)
    full = int(K * int(bl.astype(np.int64).sum()) * 2)
    for f in budgets:
        B = int(f * full)
        plan = mp.mp_plan(idx, gop, B)
        pi = mp.mp_plan_info(plan, idx)
        want = oracle.plan(K, bl, bt, len(numels), 2, oop, norm, norm, nnz, None, B,
                           blk_tensor=bt if missing else None)
        for k in ("chat", "n_sel", "n_cand", "digest"):
            assert pi[k] == want[k], (k, f)
        assert np.array_equal(pi["mask"], want["mask"]), f
        assert np.array_equal(pi["order"], want["order"]), f
        plan.free()
    idx.free()


def lognormal(rng, shape):
    return np.exp(rng.normal(-3, 2, shape))


BUDGETS = (0.0, 1e-4, 0.1, 0.5003, 0.9, 1.0)


@pytest.mark.parametrize("n_blocks,K", [(1, 1), (31, 1), (33, 1), (341, 3), (1024, 2), (1025, 2), (4097, 4),
                                        (16385, 2), (32768, 4), (32769, 4), (33000, 32)])
def test_plan_at_the_edges_of_its_launches(n_blocks, K):
    _check([256 * n_blocks - 7], 256, K, lognormal, BUDGETS if n_blocks * K < 1 << 19 else (0.3, 1.0), zero_frac=0.1)


@pytest.mark.parametrize("norms", [lambda r, s: np.ones(s), lambda r, s: np.zeros(s),
                                   lambda r, s: 2.0 ** r.integers(-3, 3, s)], ids=["equal", "zero", "powers"])
def test_plan_with_scores_that_tie(norms):
    _check([256 * 700 - 3, 5, 256 * 40], 256, 5, norms, BUDGETS)


@pytest.mark.parametrize("score_mode", [0, 1])
@pytest.mark.parametrize("missing", [0.0, 0.002])
def test_plan_with_a_long_tail_of_unequal_costs(score_mode, missing):
    rng = np.random.default_rng(3)
    numels = [int(n) for n in rng.integers(3, 700, 3000)] + [256 * 50]
    _check(numels, 256, 4, lognormal, (0.05, 0.2, 0.5, 0.777, 0.95, 0.9999), 0.05, missing, score_mode, seed=4)


def test_a_tail_that_fits_at_once():
    # one huge unit first in the order overflows the budget, thousands of small ones follow
    numels = [1 << 20] + [9] * 9000
    def norms(r, s):
        n = np.full(s, 1e-3)
        n[:, 0] = 1.0
        return n * (1 + 1e-3 * r.random(s))
    _check(numels, 1 << 20, 1, norms, (0.01, 0.05, 0.5, 1.0))


@pytest.mark.parametrize("norms", [lognormal, lambda r, s: 2.0 ** r.integers(-3, 3, s), lambda r, s: np.zeros(s)],
                         ids=["lognormal", "powers", "zero"])
@pytest.mark.parametrize("n_blocks,K", [(7, 1), (257, 2), (1023, 1), (1365, 2), (3072, 1), (1024, 3), (3073, 1)])
def test_units_ranked_by_comparison(n_blocks, K, norms):
    # up to 3,072 units; candidates fewer than units, not a multiple of 4 or 32, tensors with missing entries
    _check([256 * n_blocks - 7], 256, K, norms, (0.0, 0.3, 1.0), zero_frac=0.13, seed=n_blocks)
    _check([256 * (n_blocks - 3) - 7, 300, 5], 256, K, norms, (0.3, 1.0), missing=0.01, seed=n_blocks)


@pytest.mark.parametrize("n_blocks,K", [(1, 1), (33, 1), (700, 3), (3073, 1), (16385, 2)])
def test_plan_without_room_for_a_cluster(n_blocks, K):
    """what one cluster plans otherwise, by the cooperative grid: single units, fewer than its warps, and
    sizes of both ways of ordering; the first plan and one from the kept order"""
    class Refused:
        def __enter__(self):
            self.plan = mp.mp_plan
            def plan(*a, **k):
                mp.mp_debug_inject_fault(mp.MP_FAULT_CLUSTER, 1)
                return self.plan(*a, **k)
            mp.mp_plan = plan
        def __exit__(self, *a):
            mp.mp_plan = self.plan
            mp.mp_debug_inject_fault(mp.MP_FAULT_CLUSTER, 0)

    with Refused():
        _check([256 * n_blocks - 7], 256, K, lognormal, (0.0, 0.3, 1.0), zero_frac=0.13)
        _check([256 * n_blocks - 7, 300, 5], 256, K, lognormal, (0.3, 1.0), missing=0.01)
