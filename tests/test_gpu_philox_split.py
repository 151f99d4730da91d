"""The merge kernels' Philox4x32-10 (first two rounds shared over experts and groups) against the
oracle's, over all four counter words — group numbers above 2^32 among them, which no family
that fits a test reaches — and both key words."""
import ctypes
import os
import subprocess
import tempfile

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_split_philox_matches_the_oracle():
    from paper_2605_29489_gb300 import build

    so = os.path.join(tempfile.mkdtemp(prefix="philox_split_"), "probe.so")
    subprocess.check_call([build.nvcc(), *build.ARCH, "-std=c++17", "-O2", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                           os.path.join(HERE, "probes", "philox_split_probe.cu"), "-o", so])
    L = ctypes.CDLL(so)
    L.philox_split_probe.restype = ctypes.c_int
    L.philox_split_probe.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_uint, ctypes.c_void_p]
    rng = np.random.default_rng(11)
    n = 512
    ctr = rng.integers(0, 2 ** 32, (n, 4), dtype=np.uint64).astype(np.uint32)
    ctr[:256, 2] = rng.integers(0, 32, 256)
    ctr[:256, 3] = 0x44415245
    ctr[:64, 1] = 0
    ctr[0] = 0
    key = rng.integers(0, 2 ** 32, (n, 2), dtype=np.uint64).astype(np.uint32)
    key[:8] = 0
    d_c, d_k = (torch.from_numpy(x.view(np.int32)).cuda() for x in (ctr, key))
    out = torch.zeros(n, 4, dtype=torch.int32, device="cuda")
    assert L.philox_split_probe(d_c.data_ptr(), d_k.data_ptr(), n, out.data_ptr()) == 0
    got = out.cpu().numpy().view(np.uint32)
    for t in range(n):
        assert np.array_equal(oracle.philox4x32_10([int(x) for x in ctr[t]], [int(x) for x in key[t]]), got[t]), t
