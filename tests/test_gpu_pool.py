"""The library's device-memory pool: bounded after the handles are freed, and safe with several
threads and streams using (and freeing) handles at once."""
import threading

import numpy as np
import pytest
import torch

from test_gpu_parity import upload

pytestmark = pytest.mark.gpu

import paper_2605_29489_gb300 as mp  # noqa: E402
from paper_2605_29489_gb300 import synth  # noqa: E402


def test_unused_memory_is_bounded():
    # a TIES_MASKED catalog holds a kilobyte or more per unit: 400,000 units, several at once
    fam = synth.custom([12500 * 256], dtype=synth.BF16, block_elems=256, K=32, name="pool-bound")
    b = torch.zeros(fam.total_elems, dtype=torch.bfloat16, device="cuda")
    mf = mp.family([(0, 12500 * 256)], b, [b] * 32, 256, mp.MP_BF16, 0)
    op = mp.make_op(mp.MP_OP_TIES_MASKED, density=0.2)
    mp.mp_index_blocks(mf, op).free()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    hs = [mp.mp_index_blocks(mf, op) for _ in range(4)]
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] > 1 << 30
    for h in hs:
        h.free()
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 256 << 20


def test_threads_on_their_own_streams():
    fam = synth.custom([70001, 4096 * 40, 300], dtype=synth.BF16, block_elems=4096, K=3, active_frac=0.5, name="pool-mt")
    base, experts = fam.host_arrays()
    mf, b, ex = upload(fam, base, experts)
    ops = [mp.make_op(mp.MP_OP_TIES, density=0.2), mp.make_op(mp.MP_OP_TA, alpha=[0.3] * 3),
           mp.make_op(mp.MP_OP_DARE_TIES, drop_p=0.5, seed=3), mp.make_op(mp.MP_OP_TIES_MASKED, density=0.3)]
    B = mp.mp_budget_from_fraction(mf, 0.5)

    def merge(op, st):
        out = torch.zeros_like(b)
        st.wait_stream(torch.cuda.default_stream())
        with mp.mp_index_blocks(mf, op, stream=st) as idx, mp.mp_plan(idx, op, B, stream=st) as plan:
            with mp.mp_merge(mf, idx, plan, out, stream=st) as man:
                dig = mp.mp_manifest_info(man, 3)["digest"]
        return out, dig

    want = [merge(op, torch.cuda.Stream()) for op in ops]
    torch.cuda.synchronize()
    bad = []

    def work(k):
        st = torch.cuda.Stream()
        for r in range(25):
            out = torch.zeros_like(b)
            torch.cuda.default_stream().synchronize()
            out, dig = merge(ops[k], st)
            st.synchronize()
            if dig != want[k][1] or not torch.equal(out.view(torch.int16), want[k][0].view(torch.int16)):
                bad.append((k, r))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(len(ops))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
