"""GPU: Lloyd iterations of small fp32 problems in one launch against the chain of launches, bit for bit: one and several tiles of points per
CTA, two and four points per thread, centre counts around its groups of 16, 32 and 64, CTAs without points, empty clusters, rows of NaN."""
import pytest
import torch

pytestmark = pytest.mark.gpu

CHAIN = 128                                    # muse_test_force_paths: the chain of launches


@pytest.mark.parametrize("D,B,Hq,Hkv,N,Cq,Ck,S,T", [
    (64, 1, 1, 1, 64, 1, 2, 8, 1), (64, 1, 1, 1, 1024, 8, 16, 8, 5), (128, 1, 3, 1, 130, 15, 17, 2, 2), (64, 1, 2, 1, 999, 33, 250, 9, 1),
    (128, 1, 2, 1, 4096, 49, 128, 4, 3), (64, 2, 4, 2, 1503, 37, 90, 3, 3), (128, 1, 12, 3, 2000, 64, 80, 5, 2)])
def test_one_launch_equals_the_chain(D, B, Hq, Hkv, N, Cq, Ck, S, T):
    from paper_2509_10406_b200 import binding as mb
    from tests.gpu_util import kernels_launched
    g = torch.Generator(device="cuda").manual_seed(N + Ck)
    e = lambda *shape: torch.randn(*shape, generator=g, device="cuda")  # noqa: E731
    Q, K = e(B, Hq, N, D), e(B, Hkv, N, D)
    start = lambda h, C: torch.rand(B * h, N, generator=g, device="cuda").topk(C, dim=1).indices.to(torch.int32).view(B, h, C).contiguous()  # noqa: E731
    iq, ik = start(Hq, Cq), start(Hkv, Ck)
    ik[:, :, -1] = ik[:, :, 0]                 # of two equal centres the later is empty from the first assignment on
    if N > 500:
        K[:, :, 5:9] = float("nan")
    p = mb.make_params(B=B, Hq=Hq, Hkv=Hkv, N=N, D=D, Cq=Cq, Ck=Ck, m=1, n_blocks=S, causal=S > 1, dtype="f32", kmeans_iters=T)
    ws = torch.empty(mb.muse_workspace_bytes(p)[0], dtype=torch.uint8, device="cuda")
    got = []
    for mask in (CHAIN, 0):
        out = [torch.full((B, Hq, N), -7, dtype=torch.int32, device="cuda"), torch.full((B, Hkv, N), -7, dtype=torch.int32, device="cuda"),
               torch.zeros(B, Hq, Cq, D, device="cuda"), torch.zeros(B, Hkv, Ck, D, device="cuda")]
        mb.muse_test_force_paths(mask)
        try:
            with kernels_launched() as k:
                mb.muse_cluster(p, Q, K, iq, ik, *out, ws)
        finally:
            mb.muse_test_force_paths(0)
        assert ("k_lloyd_small" in k.names) == (mask == 0)
        assert mb.muse_status(ws) == 0
        got.append([x.view(torch.int32) for x in out])
    for a, b in zip(*got):
        assert torch.equal(a, b)
