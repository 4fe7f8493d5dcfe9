"""Calls on a stream that owns a part of the GPU's SMs (a green context):
the cooperative kernels take no more CTAs than that part holds.  Against the
oracle, bit-exact."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Resource(ctypes.Structure):  # CUdevResource; words[0]: the SM count
    _fields_ = [("type", ctypes.c_int), ("pad", ctypes.c_ubyte * 92), ("words", ctypes.c_uint * 12)]


@pytest.fixture(scope="module")
def partition_stream():
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        rc = getattr(cu, name)(*args)
        if rc != 0:
            pytest.skip(f"{name}: {rc}")

    whole, part, own = Resource(), Resource(), Resource()
    desc, green, stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    count = ctypes.c_uint(1)
    call("cuDeviceGetDevResource", 0, ctypes.byref(whole), 1)
    call("cuDevSmResourceSplitByCount", ctypes.byref(part), ctypes.byref(count), ctypes.byref(whole), None, 0, 16)
    call("cuDevResourceGenerateDesc", ctypes.byref(desc), ctypes.byref(part), 1)
    call("cuGreenCtxCreate", ctypes.byref(green), desc, 0, 1)
    call("cuGreenCtxGetDevResource", green, ctypes.byref(own), 1)
    assert 0 < own.words[0] < whole.words[0]
    call("cuGreenCtxStreamCreate", ctypes.byref(stream), green, 1, 0)
    yield stream.value
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(green)


@pytest.mark.parametrize("n", [333, 20_000, 100_003])
def test_emst_and_dendrogram(partition_stream, n):
    import paper_2207_00514_gb300 as pkg
    pts = synth.blobs(n, 3, n)
    t = torch.from_numpy(pts).cuda()
    torch.cuda.synchronize()
    edges = pkg.emst_compute(t, stream=partition_stream)
    link, parent = pkg.emst_dendrogram(edges, n, stream=partition_stream)
    torch.cuda.synchronize()
    e = pkg.edges_numpy(edges)
    assert np.array_equal(e.view(np.uint32), oracle.emst(pts).view(np.uint32))
    want_link, want_parent = oracle.dendrogram(e, n)
    assert np.array_equal(pkg.linkage_numpy(link).view(np.uint32), want_link.view(np.uint32))
    assert np.array_equal(parent.cpu().numpy().view(np.uint32), want_parent)
