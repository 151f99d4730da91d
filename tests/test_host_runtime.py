"""The library's host code on a CUDA runtime without a device (CPU).

The library's own sources are linked against `probes/fake_cudart.cpp`, where kernels do nothing, work on a
stream is done only when something waits for it, and device memory is host memory against a limit.
What the host code waits for, which allocations it makes and which launches it chooses can then be
seen without a GPU, also for what must not be tried on one: memory handed back while a kernel
may still read it, a device that is nearly full, a planner that gives up.
"""
import concurrent.futures as cf
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

import paper_2605_29489_gb300 as mp

HERE = os.path.dirname(os.path.abspath(__file__))
OOM, TIMEOUT = -3, -6
DEVICE_GB = 280


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    from paper_2605_29489_gb300 import build

    d = str(tmp_path_factory.mktemp("fake_runtime"))
    srcs = sorted(glob.glob(os.path.join(build.CSRC, "*.cu"))) + [os.path.join(HERE, "probes", "fake_cudart.cpp")]
    objs = [os.path.join(d, os.path.basename(s) + ".o") for s in srcs]
    # PTX only: nothing here is run on a device
    flags = ["-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "-O1", "-Xcompiler", "-fPIC",
             "--expt-relaxed-constexpr", "-I", build.INCLUDE, "-I", build.CSRC]
    with cf.ThreadPoolExecutor(max_workers=os.cpu_count() or 4) as ex:
        list(ex.map(lambda so: subprocess.check_call([build.nvcc(), *flags, "-c", so[0], "-o", so[1]]), zip(srcs, objs)))
    path = os.path.join(d, "libmergepipe_fake.so")
    subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic", "-o", path, *objs])
    return path


@pytest.fixture
def rt(fake_lib, monkeypatch):
    """the package's binding over the library on the fake runtime; the runtime's own controls"""
    monkeypatch.setattr(mp, "library_path", lambda: fake_lib)
    monkeypatch.setattr(mp, "_lib", None)
    L = mp.lib()
    for n in ("fake_used", "fake_pending", "fake_most_pending_at_free"):
        getattr(L, n).restype = ctypes.c_uint64
    L.fake_memory.argtypes = [ctypes.c_size_t, ctypes.c_size_t]
    L.fake_launched.argtypes = [ctypes.c_char_p]
    L.cudaDeviceSynchronize()
    L.fake_reset()
    yield L
    mp.mp_debug_inject_fault(mp.MP_FAULT_ALLOC, 0)


def family(n_blocks=64, K=3, block=4096, tail=0):
    """no data is read: the kernels do nothing"""
    buf = np.zeros(64, np.uint8)
    p = (buf.ctypes.data + 15) & ~15
    n = n_blocks * block - tail
    far = [p + 16 * n * (i + 1) for i in range(K + 1)]  # the buffers do not overlap the output
    fam = mp.family([(0, n)], p, far[:K], block, mp.MP_BF16, 0)
    fam.keep = buf
    return fam, far[K]


S1, S2 = 0x1000, 0x2000
TA = lambda K: mp.make_op(mp.MP_OP_TA, alpha=[0.5] * K)  # noqa: E731


# ---- a handle's memory goes back only when nothing reads it any more --------------------------

def test_freeing_waits_for_the_calls_that_use_the_handle(rt):
    """index and plan freed right after a merge was enqueued, on the merge's stream and on another: what
    they hold is read by kernels that have not run"""
    for plan_stream, merge_stream in ((S1, S1), (S1, S2), (S2, S1)):
        for first in ("index", "plan"):
            fam, out = family()
            idx = mp.mp_index_blocks(fam, TA(3), stream=S1)
            plan = mp.mp_plan(idx, TA(3), 1 << 20, stream=plan_stream)
            man = mp.mp_merge(fam, idx, plan, out, stream=merge_stream)
            assert rt.fake_pending() > 0
            for h in ((idx, plan) if first == "index" else (plan, idx)):
                h.free()
            assert rt.fake_most_pending_at_free() == 0, (plan_stream, merge_stream, first)
            man.free()


def test_freeing_an_index_waits_for_plans_hashes_and_validation(rt):
    fam, out = family()
    idx = mp.mp_index_blocks(fam, TA(3), stream=S1)
    plan = mp.mp_plan(idx, TA(3), 1 << 20, stream=S2)
    idx.free()
    assert rt.fake_most_pending_at_free() == 0
    plan.free()

    idx = mp.mp_index_blocks(fam, TA(3), stream=S1)
    mp.mp_index_hashes(fam, idx, stream=S2)
    plan = mp.mp_plan(idx, TA(3), 1 << 20, stream=S1)
    man = mp.mp_merge(fam, idx, plan, out, stream=S1)
    mp.mp_manifest_info(man, 3, check=False)
    mp.mp_manifest_validate(fam, idx, plan, out, man, stream=S1)
    mp.mp_manifest_validate(fam, idx, plan, out, man, stream=S2)
    plan.free()
    assert rt.fake_most_pending_at_free() == 0
    idx.free()
    man.free()
    assert rt.fake_most_pending_at_free() == 0


def test_one_index_used_by_many_merges_keeps_few_events(rt):
    """a long-lived index: calls that are done are forgotten, and with many in flight the runtime is not
    asked about all of them again for every call"""
    fam, out = family()
    idx = mp.mp_index_blocks(fam, TA(3), stream=S1)
    for _ in range(300):
        plan = mp.mp_plan(idx, TA(3), 1 << 20, stream=S1)
        man = mp.mp_merge(fam, idx, plan, out, stream=S2)
        for h in (man, plan):
            h.free()
    n = rt.fake_events()
    assert n <= 64
    plan = mp.mp_plan(idx, TA(3), 1 << 20, stream=S1)
    asked = rt.fake_queries()
    mans = [mp.mp_merge(fam, idx, plan, out, stream=S2) for _ in range(1000)]  # none of them runs
    assert rt.fake_queries() - asked <= 2 * 2 * 2000  # two handles, each asked at 16, 32, 64, ...
    used = rt.fake_used()
    idx.free()
    plan.free()
    assert rt.fake_used() < used and rt.fake_most_pending_at_free() == 0
    for m in mans:
        m.free()


# ---- a planner that gives up ------------------------------------------------------------------

def test_a_plan_that_did_not_finish_is_reported(rt):
    """the planner writes its summary to the host at its very end; one that gave up before (here: that
    did not run) is a timeout, not the plan of whatever handle had the pinned slot before"""
    fam, out = family()
    idx = mp.mp_index_blocks(fam, TA(3), stream=S1)
    for _ in range(3):  # the slot is used again and again
        plan = mp.mp_plan(idx, TA(3), 1 << 20, stream=S1)
        with pytest.raises(mp.MergePipeError) as e:
            mp.mp_plan_info(plan)
        assert e.value.status == TIMEOUT
        plan.free()
    idx.free()


# ---- TIES after masking on a device that is nearly full ---------------------------------------

UNITS = 640_000  # 20,000 blocks of 2,048 elements, 32 experts: the line of the larger histograms
LARGE, SMALL = UNITS * 640 * 4, UNITS * 256 * 4
MASKED = mp.make_op(mp.MP_OP_TIES_MASKED, density=0.2)


def _masked_catalog(rt):
    """bytes held by a catalog of TIES after masking"""
    fam, _ = family(n_blocks=20_000, K=32, block=2048)
    before = rt.fake_used()
    with mp.mp_index_blocks(fam, MASKED, stream=S1):
        return rt.fake_used() - before


def test_smaller_histograms_whenever_the_larger_ones_do_not_fit(rt):
    assert _masked_catalog(rt) > LARGE
    tables = UNITS * 12 + 20_000 * 20
    for largest in (LARGE - 1,             # not even the histograms
                    LARGE + tables // 2):  # those, but not the tables and statistics beside them
        rt.fake_memory(64 << 30, largest)
        held = _masked_catalog(rt)
        assert SMALL < held < LARGE, largest
    rt.fake_memory(SMALL, 1 << 40)  # too little for those either
    with pytest.raises(mp.MergePipeError) as e:
        _masked_catalog(rt)
    assert e.value.status == OOM


def test_an_injected_failure_is_not_taken_for_a_full_device(rt):
    mp.mp_debug_inject_fault(mp.MP_FAULT_ALLOC, 1)
    with pytest.raises(mp.MergePipeError) as e:
        _masked_catalog(rt)
    assert e.value.status == OOM and "injected" in str(e.value)
    assert _masked_catalog(rt) > LARGE


def test_larger_histograms_only_where_the_caller_keeps_nearly_all_of_the_free_memory(rt):
    """983 MB more than the smaller ones: more than a 32nd of 20 GB, less than that of 40 GB"""
    rt.fake_memory(20 << 30, 1 << 40)
    assert SMALL < _masked_catalog(rt) < LARGE
    rt.fake_memory(40 << 30, 1 << 40)
    assert _masked_catalog(rt) > LARGE
    rt.fake_memory(1 << 30, 1 << 40)  # 40,000 units: 61 MB more, as before
    fam, _ = family(n_blocks=40_000, K=1, block=2048)
    before = rt.fake_used()
    with mp.mp_index_blocks(fam, MASKED, stream=S1):
        assert rt.fake_used() - before > 40_000 * 640 * 4


# ---- the memory that the library keeps --------------------------------------------------------

def test_trim_gives_the_kept_memory_back(rt):
    fam, out = family()
    mp.mp_index_blocks(fam, TA(3), stream=S1).free()
    n = rt.fake_trims()
    mp.mp_trim()
    assert rt.fake_trims() == n + 1


# ---- a device without room for the planner's cluster ------------------------------------------

def test_planner_takes_the_grid_where_no_cluster_fits(rt):
    fam, out = family()
    idx = mp.mp_index_blocks(fam, TA(3), stream=S1)
    mp.mp_plan(idx, TA(3), 1 << 20, stream=S1).free()
    assert rt.fake_launched(b"cluster:") == 1 and rt.fake_launched(b"cooperative:") == 0
    rt.fake_cluster_room(0)
    mp.mp_plan(idx, TA(3), 1 << 20, stream=S1).free()
    assert rt.fake_launched(b"cluster:") == 1 and rt.fake_launched(b"cooperative:") == 1
    idx.free()


# ---- capture of a catalog whose block table is above the largest pinned slot ------------------

def test_a_captured_upload_keeps_its_source(rt):
    """500,000 blocks, 10 MB of table: a replay copies it in again, so the copy's source has to live as
    long as the handle; outside a capture it is done when the call returns"""
    fam, out = family(n_blocks=500_000, K=1, block=256)
    idx = mp.mp_index_blocks(fam, TA(1), stream=S1)
    assert rt.fake_copies() == 1
    idx.free()
    blocks = rt.fake_host_blocks()
    rt.fake_reset()
    rt.fake_capturing(1)
    idx = mp.mp_index_blocks(fam, TA(1), stream=S1)
    rt.fake_capturing(0)
    assert rt.fake_copies() == 0 and rt.fake_host_blocks() == blocks + 1
    idx.free()
    assert rt.fake_host_blocks() == blocks
