"""Kernels of a call that may start before the one ahead of them has ended.

Back-to-back calls on families of a few blocks, where every kernel is shorter than a launch: each
pass must give the oracle's plan and output and the same bits as the first, on the default stream and on
a stream of its own whose inputs were written just before.
"""
import numpy as np
import pytest
import torch

from test_gpu_parity import ops_for, run_case, upload

pytestmark = pytest.mark.gpu

import paper_2605_29489_gb300 as mp  # noqa: E402
from paper_2605_29489_gb300 import synth  # noqa: E402

KINDS = ("ta", "ties", "dare_ties", "avg_renorm", "ties_masked")


def _family(E):
    fam = synth.custom([3 * E + 5, 9, E, 2 * E - 8], dtype=synth.BF16, block_elems=E, K=5, active_frac=0.6,
                       name="launch-order")
    return fam, *fam.host_arrays()


@pytest.mark.parametrize("E", [512, 4096])
def test_chains_of_short_kernels(E):
    fam, base, experts = _family(E)
    run_case(fam, base, experts, KINDS, [0.3, 1.0])
    side = torch.cuda.Stream()
    for name, gop, _ in ops_for(fam.K, KINDS):
        mf, b, ex = upload(fam, base, experts)
        first = None
        for it in range(30):
            st = side if it % 3 == 0 else torch.cuda.current_stream()
            st.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(st):
                for x in ex:  # written by the kernel ahead of the call
                    x.copy_(x.clone())
                out = torch.empty_like(b)
                with mp.mp_index_blocks(mf, gop, stream=st) as idx:
                    with mp.mp_plan(idx, gop, mp.mp_budget_from_fraction(mf, 0.5), stream=st) as plan:
                        man = mp.mp_merge(mf, idx, plan, out, stream=st)
                        got = (out.view(torch.int16).cpu().numpy().copy(), mp.mp_manifest_info(man, fam.K)["digest"])
                        man.free()
            torch.cuda.current_stream().wait_stream(st)
            if first is None:
                first = got
            assert got[1] == first[1] and np.array_equal(got[0], first[0]), (name, it)
