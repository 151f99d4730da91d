"""TIES, DARE and DARE-TIES merges at the edges of their groups of fills, against the oracle.

A chunk's experts are published 4 (K <= 4) or 8 at a time: expert counts on both sides of every
group and class, chunks that select none, some and all of them, ragged tensors and partial chunks.
And a chunk that crosses element 2^35, where the mask generator's counter carries into its upper
word: the producer publishes it as two.
"""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_parity import run_case

pytestmark = pytest.mark.gpu

import paper_2605_29489_gb300 as mp  # noqa: E402
from paper_2605_29489_gb300 import synth  # noqa: E402

SHAPES = [2048 * 3 + 5, 7, 4096 * 2, 1024 + 8, 30001]


@pytest.mark.parametrize("dtype", [synth.BF16, synth.F32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("K", [1, 4, 5, 8, 9, 16, 17, 24, 25, 32])
def test_merges_at_the_edges_of_the_groups(K, dtype):
    fam = synth.custom(SHAPES, dtype=dtype, block_elems=4096, K=K, active_frac=0.7, per_expert_active=True, seed=K,
                       name="groups")
    base, experts = fam.host_arrays()
    run_case(fam, base, experts, ("ties", "dare", "dare_ties"), [0.0, 0.15, 0.6, 1.0])


@pytest.mark.parametrize("kind", ["dare", "dare_ties"])
def test_a_chunk_across_the_carry_of_the_mask_counter(kind):
    torch.cuda.empty_cache()  # what earlier tests left with torch's allocator
    if torch.cuda.mem_get_info()[0] < 160 << 30:
        pytest.skip("two buffers of 2^35 bf16 elements do not fit")
    edge, before, n = 1 << 35, 8 * 1001, 20000
    off = edge - before
    rng = np.random.default_rng(5)
    bits = lambda x: torch.from_numpy(x.astype(np.float32)).to(torch.bfloat16)  # noqa: E731
    hb, hx = bits(0.02 * rng.standard_normal(n)), bits(0.02 * rng.standard_normal(n))
    base = torch.empty(off + n, dtype=torch.bfloat16, device="cuda")
    expert = torch.empty(off + n, dtype=torch.bfloat16, device="cuda")
    base[off:].copy_(hb)
    expert[off:].copy_(hx)
    E = 16384
    fam = mp.family([(off, n)], base, [expert], E, mp.MP_BF16, 0)
    gop = mp.make_op(mp.MP_OP_DARE if kind == "dare" else mp.MP_OP_DARE_TIES, alpha=[1.0], lam=0.7, drop_p=0.5, seed=9)
    oop = oracle.Op(oracle.DARE if kind == "dare" else oracle.DARE_TIES, 1, alpha=[1.0], lam=0.7, drop_p=0.5, seed=9)
    with mp.mp_index_blocks(fam, gop) as idx, mp.mp_plan(idx, gop, 2 * n) as plan:
        with mp.mp_merge_touched(fam, idx, plan, base) as man:  # in place
            assert mp.mp_manifest_info(man, 1)["realized_total"] == 2 * n
        got = base[off:].cpu().view(torch.int16).numpy().view(np.uint16)
    raw = lambda t: t.view(torch.int16).numpy().view(np.uint16)  # noqa: E731
    want = np.concatenate([oracle.merge_block(synth.BF16, off + s, raw(hb)[s:s + E], [raw(hx)[s:s + E]], 1, oop)
                           for s in range(0, n, E)])
    del fam, base, expert
    torch.cuda.empty_cache()
    assert np.array_equal(got, want)


@pytest.mark.parametrize("K", [3, 6, 11])
@pytest.mark.parametrize("n_blocks", [150, 152 * 3 * 8 + 5, 152 * 4 * 16 - 1, 152 * 4 * 24 + 9])
def test_chunks_taken_one_two_and_three_at_a_time(n_blocks, K):
    """the number of chunks of a grab follows the size of the merge (one chunk per block here)"""
    fam = synth.custom([n_blocks * 512 - 3, 77], dtype=synth.BF16, block_elems=512, K=K, active_frac=0.5,
                       name=f"grabs-{n_blocks}")
    base, experts = fam.host_arrays()
    run_case(fam, base, experts, ("ta", "ties", "dare", "avg_renorm", "dare_ties"), [0.4])


@pytest.mark.parametrize("K", [3, 6, 11])
def test_long_runs_of_chunks_that_select_no_expert(K):
    """blocks that differ from the base 12 blocks apart, so that between two of them a CTA's ring is
    held by one-slot groups only: every group entry is then outstanding, and the entry just released
    is the one published next.  Repeated, because what can go wrong there depends on timing."""
    E, nb = 65536, 733
    n = nb * E - 1001
    g = torch.Generator(device="cuda").manual_seed(K)
    base = torch.randn(n, generator=g, device="cuda").mul_(0.02).to(torch.bfloat16)
    experts = [base.clone() for _ in range(K)]
    active = sorted({*range(5, nb, 12), nb - 1})
    for i, x in enumerate(experts):
        for b in active[i % 2::2] if i else active:
            v = x[b * E:(b + 1) * E]
            v.copy_((v.float() + 1e-3 * torch.randn(v.numel(), generator=g, device="cuda")).to(torch.bfloat16))
    fam = mp.family([(0, n)], base, experts, E, mp.MP_BF16, 0)
    raw = lambda t: t.view(torch.int16).cpu().numpy().view(np.uint16)  # noqa: E731
    untouched = (base.float() + 0.0).to(torch.bfloat16)  # M_0 plus the zero that the operator adds
    kw = dict(lam=0.8, density=0.02, drop_p=0.5, seed=3, alpha=[1.0 / K] * K)
    for gk, ok in [(mp.MP_OP_TIES, oracle.TIES), (mp.MP_OP_DARE, oracle.DARE), (mp.MP_OP_DARE_TIES, oracle.DARE_TIES)]:
        gop, oop = mp.make_op(gk, **kw), oracle.Op(ok, K, **kw)
        with mp.mp_index_blocks(fam, gop) as idx, mp.mp_plan(idx, gop, mp.mp_budget_from_fraction(fam, 1.0)) as plan:
            pi = mp.mp_plan_info(plan, idx)
            tau = mp.mp_index_stats(idx)[3][:, 0] if gk == mp.MP_OP_TIES else None
            want = untouched.clone()
            for b in np.nonzero(pi["mask"])[0]:
                s = slice(int(b) * E, min((int(b) + 1) * E, n))
                w = oracle.merge_block(synth.BF16, s.start, raw(base[s]), [raw(x[s]) for x in experts],
                                       int(pi["mask"][b]), oop, tau)
                want[s].copy_(torch.from_numpy(w.view(np.int16)).view(torch.bfloat16))
            for it in range(10):
                out = torch.full_like(base, float("nan"))
                with mp.mp_merge(fam, idx, plan, out) as man:
                    assert mp.mp_manifest_info(man, K)["realized_total"] == pi["chat"], (gk, it)
                assert torch.equal(out.view(torch.int16), want.view(torch.int16)), (gk, it)
