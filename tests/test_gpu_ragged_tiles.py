"""GPU: the tensor-core far-field and key-side kernels at cluster counts that no tile divides, and both sides of the
streaming clustering in one call against each side alone."""
import numpy as np
import pytest
import torch

from tests import test_gpu_k2
from tests.gpu_util import kernels_launched, to_np
from tests.test_gpu_backward import _backward_parity, _backward_parity_run
from tests.test_gpu_cluster import CASES
from tests.test_gpu_forward import TC_BWD_KERNELS, TC_FWD_KERNELS, _forward_parity, _forward_parity_run

pytestmark = pytest.mark.gpu

RAGGED = [("d64", 5, 1, 1, 3), ("d64", 130, 127, 5, 4), ("d128", 9, 129, 8, 3), ("d128", 37, 300, 16, 4), ("d128", 3, 1100, 8, 3)]


@pytest.mark.parametrize("base,Cq,Ck,m,S", RAGGED)
def test_forward_at_ragged_cluster_counts(base, Cq, Ck, m, S):
    w = CASES[base].with_(Hq=2, Hkv=1, N=510 * S, S=S, Cq=Cq, Ck=Ck, m=m, components=64)
    _forward_parity(w, 128.0, expect_kernels=TC_FWD_KERNELS)


@pytest.mark.parametrize("base,Cq,Ck,m,S", RAGGED)
def test_backward_at_ragged_cluster_counts(base, Cq, Ck, m, S):
    w = CASES[base].with_(Hq=2, Hkv=1, N=510 * S, S=S, Cq=Cq, Ck=Ck, m=m, components=64)
    _backward_parity(w, 128.0, expect_kernels=TC_BWD_KERNELS)


@pytest.mark.parametrize("Hq,Hkv,D,Cq,Ck,cap", [(2, 1, 64, 20, 600, 1.25), (4, 4, 128, 130, 40, 1.5), (1, 1, 64, 64, 33, 4.0)])
def test_streaming_both_sides_at_once_equals_each_side_alone(Hq, Hkv, D, Cq, Ck, cap):
    from paper_2509_10406_b200 import binding as mb
    N, S = 4000, 4
    g = torch.Generator(device="cuda").manual_seed(Cq)
    Q, K = (torch.randn(1, h, N, D, generator=g, device="cuda").bfloat16() for h in (Hq, Hkv))
    p = mb.make_params(B=1, Hq=Hq, Hkv=Hkv, N=N, D=D, Cq=Cq, Ck=Ck, m=0, n_blocks=S, seed=11)
    e = lambda *s, dt=torch.float32: torch.empty(*s, dtype=dt, device="cuda")  # noqa: E731
    ws = e(mb.muse_stream_workspace_bytes(p), dt=torch.uint8)
    both = [e(1, Hq, N, dt=torch.int32), e(1, Hkv, N, dt=torch.int32), e(1, Hq, Cq, D), e(1, Hkv, Ck, D)]
    mb.muse_cluster_streaming(p, Q, K, *both, ws, cap_factor=cap)
    torch.cuda.synchronize()
    assert mb.muse_status(ws) == 0
    for side, X, H, C, assign, cen in ((0, Q, Hq, Cq, both[0], both[2]), (1, K, Hkv, Ck, both[1], both[3])):
        tot, cnt, c1, a1 = e(1, H, C, D), e(1, H, C), e(1, H, C, D), e(1, H, N, dt=torch.int32)
        mb.muse_stream_kmeans(p, X, side, tot, cnt, c1, ws)
        mb.muse_balanced_assign(p, X, side, c1, a1, ws, cap_factor=cap)
        torch.cuda.synchronize()
        assert np.array_equal(to_np(c1), to_np(cen)) and np.array_equal(to_np(a1), to_np(assign))
        size = np.bincount(to_np(a1)[0, 0, :N // S], minlength=C)
        assert size.sum() == N // S and size.max() <= max(1, int(np.ceil(cap * (N // S) / C)))


@pytest.mark.parametrize("base,Ck,m,two_kernels", [("d64", 7, 3, True), ("d64", 8, 3, True), ("d64", 2, 2, True), ("d64", 12, 3, True),
                                                   ("d64", 13, 3, False), ("d64", 20, 11, True), ("d64", 21, 11, False), ("d128", 15, 3, True),
                                                   ("d128", 16, 3, True), ("d128", 25, 3, True), ("d128", 26, 3, False)])
def test_retrieval_on_both_sides_of_the_cluster_length_rule(base, Ck, m, two_kernels):
    """2040 keys: below 80 (D = 128) or 100 keys a cluster, or 160 with few pairs, the fused backward kernel; below 128 or 256 the forward
    kernel with resident keys."""
    w = CASES[base].with_(Hq=2, Hkv=1, N=2040, S=4, Cq=9, Ck=Ck, m=m, components=64)
    with kernels_launched() as rec:
        _backward_parity_run(w, 128.0)
    assert "k_ret_bwd_pairs_tc" in rec.names and ("k_ret_bwd_dq" in rec.names) == two_kernels
    streamed = 2040 // Ck >= (128 if w.D == 128 else 256)
    assert {n for n in rec.names if n.startswith(("k_ret_fwd_pairs_tc/", "k_ret_bwd_pairs_tc/"))} == {
        "k_ret_fwd_pairs_tc/" + ("k_ret_fwd_long" if streamed else "k_ret_fwd_pairs_tc"),
        "k_ret_bwd_pairs_tc/" + ("k_ret_bwd_dkdv" if two_kernels else "k_ret_bwd_sweeps")}, sorted(rec.names)


@pytest.mark.parametrize("base,Cq,Ck,m,S,k2", [("d64", 5, 9, 4, 10, 1), ("d64", 3, 40, 33, 3, 1), ("d128", 7, 10, 5, 12, 2), ("d128", 1, 6, 6, 2, 1)])
def test_near_field_backward_over_groups_of_blocks(monkeypatch, base, Cq, Ck, m, S, k2):
    """More earlier blocks than one group of the kernel (8 at D = 64, 4 at D = 128), more than 32 slots, one earlier block."""
    w = CASES[base].with_(Hq=2, Hkv=1, N=330 * S, S=S, Cq=Cq, Ck=Ck, m=m, components=64)
    monkeypatch.setitem(test_gpu_k2.K2_CASES, "groups", w)
    test_gpu_k2.test_two_level_backward_matches_oracle("groups", k2, True, 4)


@pytest.mark.parametrize("base,Cq,Ck,m", [("d64", 2, 256, 16), ("d64", 3, 128, 9), ("d64", 5, 2, 1), ("d128", 2, 256, 8), ("d128", 3, 127, 16), ("d64", 4, 256, 17)])
def test_selection_and_far_field_of_few_clusters(base, Cq, Ck, m):
    """Lists of 8 and 16 (and one more, which another kernel takes), one and two tiles of clusters, several passes over a segment."""
    w = CASES[base].with_(Hq=2, Hkv=1, N=1020, S=4, Cq=Cq, Ck=Ck, m=m, components=64)
    with kernels_launched() as rec:
        _forward_parity_run(w, 128.0)
    assert TC_FWD_KERNELS <= rec.names, sorted(rec.names)
    # (once with the GPU's selection, once with the oracle's: a given selection may be of any length)
    assert {n for n in rec.names if n.startswith("k_far_fwd_tc/")} == (
        {"k_far_fwd_tc/k_far_fwd_small"} | ({"k_far_fwd_tc/k_far_fwd_tc"} if m > 16 else set())), sorted(rec.names)


@pytest.mark.parametrize("base,Cq,Ck,m", [("d64", 1, 128, 20), ("d64", 2, 129, 33), ("d128", 1, 128, 33), ("d128", 3, 90, 4)])
def test_far_field_and_key_side_backward_over_long_segments(base, Cq, Ck, m):
    """Segments of several sweeps over one tile of clusters (accumulated on chip) and over two (added in memory), and selections
    longer than the far-field backward keeps in flight."""
    w = CASES[base].with_(Hq=2, Hkv=1, N=1020, S=4, Cq=Cq, Ck=Ck, m=m, components=64)
    _backward_parity(w, 128.0, expect_kernels=TC_BWD_KERNELS)
