"""GPU: retrieval forward of clusters of very uneven sizes, where the short ones and the long ones of one index go to different kernels
(D = 128, four million pairs), against the library's streamed FFMA retrieval.  O is a bf16 number made of bf16 weights on both sides: two
roundings, 2^-7 of the scale; LSE is fp32."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("largest", [3000, 161, 160])
def test_short_and_long_clusters_of_one_index(largest):
    from paper_2509_10406_b200 import binding as mb
    from tests.gpu_util import kernels_launched
    B, Hq, Hkv, N, D, Cq, Ck, m = 1, 4, 2, 32768, 128, 16, 512, 32
    g = torch.Generator(device="cuda").manual_seed(largest)
    e = lambda h, n: torch.randn(B, h, n, D, generator=g, device="cuda")  # noqa: E731
    # cluster sizes: a few of `largest` keys, one of none, the rest even
    big = min(20, N // (2 * largest)) if largest > 1000 else 100
    a = torch.empty(Hkv, N, dtype=torch.int32, device="cuda")
    for h in range(Hkv):
        rest = torch.randint(big + 1, Ck, (N - big * largest,), generator=g, device="cuda", dtype=torch.int32)
        a[h] = torch.cat([torch.arange(big, device="cuda", dtype=torch.int32).repeat_interleave(largest), rest])[torch.randperm(N, generator=g, device="cuda")]
    Q, K, V = (e(Hq, N) * 3).to(torch.bfloat16), e(Hkv, N).to(torch.bfloat16), e(Hkv, N).to(torch.bfloat16)
    p = mb.make_params(B=B, Hq=Hq, Hkv=Hkv, N=N, D=D, Cq=Cq, Ck=Ck, m=m)
    a_q = torch.randint(0, Cq, (B, Hq, N), generator=g, device="cuda", dtype=torch.int32)
    # every query retrieves some of the largest clusters and random others
    sel = torch.rand(B, Hq, N, Ck, generator=g, device="cuda").topk(m, dim=-1).indices.to(torch.int32)
    sel[..., :8] = torch.arange(8, device="cuda")
    sel[..., 8:][sel[..., 8:] < 8] = -1
    qbar = e(Hq, Cq)
    got = []
    for mask in (8, 0):
        buf = mb.MuseBuffers(p, backward=False)
        mb.muse_test_force_paths(mask)
        try:
            mb.muse_summarize(p, K, V, a.view(B, Hkv, N), qbar, buf.off_k, buf.perm_k, buf.summaries, buf.ws)
            with kernels_launched() as k:
                mb.muse_attn_fwd(p, Q, K, V, a_q, qbar, buf.off_k, buf.perm_k, buf.summaries, sel, buf.O, buf.LSE, buf.sel, buf.ws)
        finally:
            mb.muse_test_force_paths(0)
        assert mb.muse_status(buf.ws) == 0
        assert mask or {"k_ret_fwd_pairs_tc/k_ret_fwd_pairs_tc", "k_ret_fwd_pairs_tc/k_ret_fwd_long"} <= set(k.names)
        got.append((buf.O.float(), buf.LSE.clone()))
    (o0, l0), (o1, l1) = got
    assert (o1 - o0).abs().max() <= 2.0 ** -7 * o0.abs().max()
    assert (l1 - l0).abs().max() <= 2.0 ** -8          # (probabilities are summed as rounded to bf16 on one side)
