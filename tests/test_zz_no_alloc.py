"""muse_cluster_noalloc (clustering on the library's built-in scratch array, for callers that
cannot allocate device memory) must reproduce muse_cluster, call after call.

The file name sorts last on purpose: if this add-on fails, a run that stops at the first
failure has already exercised every other test."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2509_10406_b200 import workloads as wl
from tests.gpu_util import Case, to_dev, to_np


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["tiny", "bf16"])
def test_noalloc_cluster_matches_workspace_version_twice(name):
    from paper_2509_10406_b200 import binding as mb
    w = wl.WORKLOADS["tiny"] if name == "tiny" else wl.WORKLOADS["small"].with_(B=1, Hq=4, Hkv=2, N=4096, Cq=32, Ck=64, components=64)
    c = Case(w, gain=128.0, cluster=False)
    Q, K, V, _ = c.dev()
    iq, ik = to_dev(c.init_q, "i"), to_dev(c.init_k, "i")
    p = c.params()
    assert mb.muse_workspace_bytes(p)[0] <= mb.muse_cluster_noalloc_max_bytes()
    ref = mb.MuseBuffers(p, backward=False)
    mb.muse_cluster(p, Q, K, iq, ik, ref.assign_q, ref.assign_k, ref.qbar, ref.kcent, ref.ws)
    torch.cuda.synchronize()
    exp = [to_np(x).copy() for x in (ref.assign_q, ref.assign_k, ref.qbar, ref.kcent)]
    for call in range(2):                       # the second call finds the first call's leftovers in the scratch
        out = mb.MuseBuffers(p, backward=False)
        for t in (out.assign_q, out.assign_k):
            t.fill_(-7)
        torch.cuda.synchronize()
        # bytes the DRIVER reports free on the device: unlike torch's own counter, this would also see an
        # allocation made inside the library.  The first call may load the library's device image (that is
        # when its 32 MiB are reserved), so the comparison is made on the second call.
        free_before = torch.cuda.mem_get_info()[0]
        mb.muse_cluster_noalloc(p, Q, K, iq, ik, out.assign_q, out.assign_k, out.qbar, out.kcent)
        torch.cuda.synchronize()
        if call == 1:
            assert torch.cuda.mem_get_info()[0] >= free_before
        assert mb.muse_cluster_noalloc_status() == 0
        got = [to_np(x) for x in (out.assign_q, out.assign_k, out.qbar, out.kcent)]
        assert np.array_equal(got[0], exp[0]) and np.array_equal(got[1], exp[1]), f"assignments differ on call {call}"
        assert np.abs(got[2] - exp[2]).max() <= 1e-6 * np.abs(exp[2]).max()
        assert np.abs(got[3] - exp[3]).max() <= 1e-6 * np.abs(exp[3]).max()


@pytest.mark.gpu
def test_noalloc_rejects_problems_larger_than_its_scratch():
    from paper_2509_10406_b200 import binding as mb
    p = mb.make_params(B=4, Hq=32, Hkv=32, N=131072, D=128, Cq=512, Ck=2048, m=32)
    assert mb.muse_workspace_bytes(p)[0] > mb.muse_cluster_noalloc_max_bytes()
    one = torch.zeros(64, device="cuda")
    rc = mb.lib().muse_cluster_noalloc(ctypes.byref(p), *([ctypes.c_void_p(one.data_ptr())] * 8), None)
    assert rc == -3 and b"workspace" in mb.lib().muse_strerror(rc)


# a problem whose sides fit the built-in scratch one at a time, not together
SPLIT = dict(B=8, Hq=64, Hkv=64, N=8192, D=64, Cq=64, Ck=32, m=0, kmeans_iters=1)


def test_noalloc_checks_every_argument_before_it_does_anything():
    """Needs no GPU: a call with an invalid argument on either side is refused before the built-in array is looked up, also where the
    sides would run one after the other."""
    from paper_2509_10406_b200 import binding as mb
    fake, odd, z = ctypes.c_void_p(4096), ctypes.c_void_p(4100), ctypes.c_void_p(0)
    for kw in (SPLIT, dict(SPLIT, B=1, Hq=1, Hkv=1)):
        p = mb.make_params(**kw)
        assert (mb.muse_workspace_bytes(p)[0] > mb.muse_cluster_noalloc_max_bytes()) == (kw is SPLIT)
        good = [fake] * 8                          # Q, K, init_q, init_k, assign_q, assign_k, qbar, kcent
        for at in range(2, 8):
            assert mb.lib().muse_cluster_noalloc(ctypes.byref(p), *good[:at], z, *good[at + 1:], None) == -1
        for at in (0, 1, 6, 7):
            assert mb.lib().muse_cluster_noalloc(ctypes.byref(p), *good[:at], odd, *good[at + 1:], None) == -1
        assert mb.lib().muse_cluster_noalloc(ctypes.byref(p), z, z, *good[2:], None) == -1


def _split_problem(mb, init_mode):
    p = mb.make_params(**SPLIT, init_mode=init_mode, seed=5)
    g = torch.Generator(device="cuda").manual_seed(5)
    Q, K = (torch.randn(8, 64, 8192, 64, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    e = lambda C: (torch.empty(8, 64, 8192, dtype=torch.int32, device="cuda"), torch.empty(8, 64, C, 64, device="cuda"))  # noqa: E731
    (aq, qb), (ak, kc) = e(64), e(32)
    return p, Q, K, [aq, ak, qb, kc]


@pytest.mark.gpu
@pytest.mark.parametrize("init_mode", [1, 3])       # strided, k-means++
def test_noalloc_takes_the_sides_in_turn_where_they_do_not_fit_together(init_mode):
    from paper_2509_10406_b200 import binding as mb
    p, Q, K, out = _split_problem(mb, init_mode)
    ref = [torch.empty_like(x) for x in out]
    ws = torch.empty(mb.muse_workspace_bytes(p)[0], dtype=torch.uint8, device="cuda")
    mb.muse_cluster(p, Q, K, None, None, *ref, ws)
    mb.muse_cluster_noalloc(p, Q, K, None, None, *out)
    torch.cuda.synchronize()
    assert mb.muse_status(ws) == 0 and mb.muse_cluster_noalloc_status() == 0
    assert torch.equal(out[0], ref[0]) and torch.equal(out[1], ref[1])
    for x, y in zip(out[2:], ref[2:]):
        assert (x - y).abs().max() <= 1e-6 * y.abs().max()


def _status_clears(call):
    """Captures `call` and counts what clears the status words: memsets of their 256 bytes, and starting kernels that are handed them."""
    from cuda.bindings import driver as cu
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    graph = cu.CUgraph(g.raw_cuda_graph())
    err, _, n = cu.cuGraphGetNodes(graph)
    err, nodes, n = cu.cuGraphGetNodes(graph, n)
    memsets = kernels = starts = 0
    for node in nodes:
        kind = cu.cuGraphNodeGetType(node)[1]
        if kind == cu.CUgraphNodeType.CU_GRAPH_NODE_TYPE_MEMSET:
            pr = cu.cuGraphMemsetNodeGetParams(node)[1]
            memsets += pr.width * pr.elementSize * max(pr.height, 1) == 256
        elif kind == cu.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            pr = cu.cuGraphKernelNodeGetParams(node)[1]
            if b"k_init_centres" in cu.cuFuncGetName(pr.func)[1]:          # (sides, D, init_mode, seed, words to clear)
                starts += 1
                at = ctypes.cast(int(pr.kernelParams), ctypes.POINTER(ctypes.c_void_p))[4]
                kernels += ctypes.c_void_p.from_address(at).value is not None
    g.reset()
    return starts, memsets + kernels


@pytest.mark.gpu
def test_noalloc_clears_the_status_words_once_per_call():
    """... so that a code reported early in a call is still there at its end."""
    from paper_2509_10406_b200 import binding as mb
    for init_mode in (1, 3):
        p, Q, K, out = _split_problem(mb, init_mode)
        call = lambda: mb.muse_cluster_noalloc(p, Q, K, None, None, *out)  # noqa: E731
        call()
        torch.cuda.synchronize()
        assert _status_clears(call) == (2, 1)


@pytest.mark.gpu
def test_streaming_and_lloyd_clear_the_status_words_once_per_call():
    from paper_2509_10406_b200 import binding as mb
    p = mb.make_params(B=1, Hq=2, Hkv=2, N=2048, D=64, Cq=24, Ck=40, m=0, seed=1)
    Q, K = (torch.randn(1, 2, 2048, 64, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    buf = mb.MuseBuffers(p, backward=False)
    ws = torch.empty(mb.muse_stream_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    call = lambda: mb.muse_cluster_streaming(p, Q, K, buf.assign_q, buf.assign_k, buf.qbar, buf.kcent, ws)  # noqa: E731
    call()
    torch.cuda.synchronize()
    assert _status_clears(call) == (1, 1)
    call = lambda: mb.muse_cluster(p, Q, K, buf.sel, buf.sel, buf.assign_q, buf.assign_k, buf.qbar, buf.kcent, buf.ws)  # noqa: E731
    p.init_mode = 1
    call()
    torch.cuda.synchronize()
    assert _status_clears(call) == (1, 1)
