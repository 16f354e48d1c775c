"""GPU: far field, forward, of short query segments (at most 28 queries a segment on average and 128 clusters, where a pass holds half
the queries and each has twice the threads): segments of none to several passes, selections of one to sixteen, cluster counts around a tile
and a thread's share, against the library's FFMA kernel.  O is made of bf16 weights: two roundings, 2^-7 of its scale, 2^-8 in the
log-sum-exp.  Two evaluations of a score differ by 2^-18 of its size; of some hundred scores within +-5 the m-th and the next lie that
close for 1e-4 of the queries, which may select either: at most 1e-3 do, and the others are compared."""
import pytest
import torch

pytestmark = pytest.mark.gpu

FAR_SIMT = 2                                   # muse_test_force_paths: the FFMA far field


@pytest.mark.parametrize("D,Cq,Ck,S,m,causal", [
    (64, 40, 1, 4, 1, True), (64, 40, 9, 5, 8, True), (64, 33, 127, 3, 16, True), (64, 64, 128, 8, 0, True), (64, 90, 120, 6, 9, True),
    (64, 128, 64, 1, 5, False), (128, 40, 17, 4, 9, True), (128, 48, 128, 5, 8, True), (128, 70, 100, 4, 16, True)])
def test_short_segments_match_the_ffma_kernel(D, Cq, Ck, S, m, causal):
    _compare(D, Cq, Ck, S, m, causal, S * Cq * 20, "k_far_fwd_tc/k_far_fwd_small")


@pytest.mark.parametrize("D,Cq,Ck,S,m", [
    (64, 12, 257, 3, 20), (64, 8, 1024, 2, 32), (64, 10, 1100, 2, 17), (64, 6, 2048, 2, 40), (128, 12, 300, 3, 33), (128, 9, 640, 2, 20),
    (128, 8, 1152, 2, 64), (128, 10, 1500, 2, 8), (128, 6, 2048, 2, 32)])
def test_many_clusters_match_the_ffma_kernel(D, Cq, Ck, S, m):
    """The kernel for more than 256 clusters, or longer selections: nu units that come through few and many places, passes of 32 and 64
    queries, one to three of them."""
    _compare(D, Cq, Ck, S, m, True, S * Cq * 60, "k_far_fwd_tc/k_far_fwd_tc")


def _compare(D, Cq, Ck, S, m, causal, N, kernel):
    from paper_2509_10406_b200 import binding as mb
    from tests.gpu_util import kernels_launched
    N = max(N, -(-Ck // S) * S)
    B, Hq, Hkv = 1, 4, 2
    g = torch.Generator(device="cuda").manual_seed(N + Ck)
    e = lambda h, n: torch.randn(B, h, n, D, generator=g, device="cuda")  # noqa: E731
    Q, K, V = (e(Hq, N) * 2).to(torch.bfloat16), e(Hkv, N).to(torch.bfloat16), e(Hkv, N).to(torch.bfloat16)
    p = mb.make_params(B=B, Hq=Hq, Hkv=Hkv, N=N, D=D, Cq=Cq, Ck=Ck, m=min(m, Ck), n_blocks=S, causal=causal)
    a_k = torch.randint(0, Ck, (B, Hkv, N), generator=g, device="cuda", dtype=torch.int32)
    u = torch.rand(B, Hq, N, generator=g, device="cuda")
    a_q = (u * u * Cq).to(torch.int32).clamp_(max=Cq - 1)                     # uneven: the first clusters take several passes
    a_q[a_q == 3] = 2                                                         # and one has no query
    qbar = 0.7 * e(Hq, Cq)
    got = []
    for mask in (FAR_SIMT, 0):
        buf = mb.MuseBuffers(p, backward=False)
        mb.muse_summarize(p, K, V, a_k, qbar, buf.off_k, buf.perm_k, buf.summaries, buf.ws)
        mb.muse_test_force_paths(mask)
        try:
            with kernels_launched() as k:
                mb.muse_attn_fwd(p, Q, K, V, a_q, qbar, buf.off_k, buf.perm_k, buf.summaries, None, buf.O, buf.LSE, buf.sel, buf.ws)
        finally:
            mb.muse_test_force_paths(0)
        assert mb.muse_status(buf.ws) == 0
        assert (kernel in k.names) == (mask == 0)
        got.append((buf.sel[..., :min(m, Ck)].sort(dim=-1).values.clone(), buf.O.float(), buf.LSE.clone()))
    (s0, o0, l0), (s1, o1, l1) = got
    same = (s0 == s1).all(dim=-1)
    assert (~same).float().mean() <= 1e-3
    assert (o1 - o0)[same].abs().max() <= 2.0 ** -7 * o0.abs().max()
    assert (l1 - l0)[same].abs().max() <= 2.0 ** -8
