"""GPU: the one-launch bucket sort and the persistent tensor-core assignment at the edges of their tiles and rules:
spatial blocks shared by several CTAs, one CTA per block, several blocks per CTA; centre counts around a tile, resident
in the ring and streamed; one and two point tiles per unit; points that no tile divides."""
import numpy as np
import pytest
import torch

from oracle import muse_oracle as orc
from tests.gpu_util import to_np

pytestmark = pytest.mark.gpu


def _mb():
    from paper_2509_10406_b200 import binding as mb
    return mb


@pytest.mark.parametrize("S,N,C", [(1, 77, 1), (1, 4096, 130), (3, 999, 7), (4, 1024, 40), (5, 2005, 64), (8, 64, 16),
                                   (9, 1053, 33), (16, 4096, 100), (8, 5000, 2049)])
def test_bucket_sort_shapes(S, N, C):
    mb = _mb()
    rng = np.random.default_rng(S * 1000 + C)
    P, D = 3, 64
    a = np.minimum(rng.integers(0, C, (1, P, N)), rng.integers(0, C, (1, P, N))).astype(np.int32)     # uneven bucket sizes
    p = mb.make_params(B=1, Hq=P, Hkv=P, N=N, D=D, Cq=1, Ck=C, m=0, n_blocks=S)
    buf = mb.MuseBuffers(p, backward=False)
    K = torch.zeros(1, P, N, D, dtype=torch.bfloat16, device="cuda")
    mb.muse_summarize(p, K, K, torch.from_numpy(a).cuda(), torch.zeros(1, P, 1, D, device="cuda"), buf.off_k, buf.perm_k, buf.summaries, buf.ws)
    torch.cuda.synchronize()
    off, perm = to_np(buf.off_k), to_np(buf.perm_k)
    for h in range(P):
        key = a[0, h].astype(np.int64) * S + np.arange(N) // (N // S)
        assert np.array_equal(perm[0, h], np.argsort(key, kind="stable"))
        assert np.array_equal(off[0, h], np.concatenate([[0], np.cumsum(np.bincount(key, minlength=C * S))]))


@pytest.mark.parametrize("D,heads,N,Cq,Ck", [(64, 1, 130, 1, 127), (64, 2, 1000, 128, 129), (64, 4, 9601, 512, 513), (128, 1, 129, 3, 128),
                                            (128, 2, 1000, 129, 300), (128, 4, 9601, 128, 257)])
def test_assignment_at_tile_edges(D, heads, N, Cq, Ck):
    mb = _mb()
    g = torch.Generator(device="cuda").manual_seed(N + Ck)
    Q, K = (torch.randn(1, heads, N, D, generator=g, device="cuda").bfloat16() for _ in range(2))
    p = mb.make_params(B=1, Hq=heads, Hkv=heads, N=N, D=D, Cq=Cq, Ck=Ck, m=0, n_blocks=1, kmeans_iters=0, init_mode=mb.MUSE_INIT_CENTRES)
    buf = mb.MuseBuffers(p, backward=False)
    buf.qbar.copy_(torch.randn(buf.qbar.shape, generator=g, device="cuda") * 0.5)
    buf.kcent.copy_(torch.randn(buf.kcent.shape, generator=g, device="cuda") * 0.5)
    mb.muse_cluster(p, Q, K, None, None, buf.assign_q, buf.assign_k, buf.qbar, buf.kcent, buf.ws)
    torch.cuda.synchronize()
    assert mb.muse_status(buf.ws) == 0
    for X, a, c in ((Q, buf.assign_q, buf.qbar), (K, buf.assign_k, buf.kcent)):
        for h in range(heads):
            x, cen, got = to_np(X)[0, h].astype(np.float64), to_np(c)[0, h].astype(np.float64), to_np(a)[0, h]
            bad = np.nonzero(orc.assign_nearest(x, cen) != got)[0]
            assert bad.size <= 1e-3 * N and (bad.size == 0 or orc.assignment_gaps(x[bad], cen).max() < 1e-4)
