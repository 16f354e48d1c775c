"""GPU: Lloyd iterations of small bf16 problems in one launch against the chain of launches, bit for bit, at the edges of its tiles and
rules: one point tile per CTA and several per ring stage, CTAs without points or without centres, one and two tiles of centres, rows past
the last centre, empty clusters, duplicate start points, rows of NaN, blocks of one point, one to sixteen CTAs per problem."""
import pytest
import torch

pytestmark = pytest.mark.gpu

CHAIN = 128                                    # muse_test_force_paths: the chain of launches


@pytest.mark.parametrize("D,B,Hq,Hkv,N,Cq,Ck,S,T", [
    (64, 1, 1, 1, 64, 1, 2, 8, 1), (128, 1, 3, 1, 130, 3, 129, 2, 2), (64, 1, 2, 1, 999, 17, 250, 9, 1), (128, 1, 10, 10, 1024, 8, 128, 4, 3),
    (64, 3, 4, 4, 5005, 37, 90, 7, 3), (64, 2, 24, 24, 1024, 32, 64, 1, 3), (128, 1, 16, 16, 8192, 64, 128, 8, 2), (64, 1, 64, 64, 4096, 16, 240, 8, 2),
    (64, 1, 1, 1, 16384, 32, 64, 16, 2), (64, 1, 5, 5, 16, 4, 4, 16, 3)])
def test_one_launch_equals_the_chain(D, B, Hq, Hkv, N, Cq, Ck, S, T):
    from paper_2509_10406_b200 import binding as mb
    from tests.gpu_util import kernels_launched
    g = torch.Generator(device="cuda").manual_seed(N + Ck)
    e = lambda *shape: torch.randn(*shape, generator=g, device="cuda")  # noqa: E731
    X = {h: (e(B, h, 40, D)[:, :, torch.randint(0, 40, (N,), generator=g, device="cuda")] + 0.5 * e(B, h, N, D)).to(torch.bfloat16) for h in {Hq, Hkv}}
    Q, K = X[Hq], X[Hkv].clone()
    start = lambda h, C: torch.rand(B * h, N, generator=g, device="cuda").topk(C, dim=1).indices.to(torch.int32).view(B, h, C).contiguous()  # noqa: E731
    iq, ik = start(Hq, Cq), start(Hkv, Ck)
    ik[:, :, -1] = ik[:, :, 0]                 # of two equal centres the later is empty from the first assignment on
    if N > 500:
        K[:, :, 5:9] = float("nan")            # (cluster 0, whose centre is NaN from then on)
    p = mb.make_params(B=B, Hq=Hq, Hkv=Hkv, N=N, D=D, Cq=Cq, Ck=Ck, m=1, n_blocks=S, causal=S > 1, kmeans_iters=T)
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
