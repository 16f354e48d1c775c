"""GPU parity with more spatial blocks than a 32-bit word has bits (more than 32 summary planes) and than the kernels keep bucket
offsets for in shared memory (72)."""
import numpy as np
import pytest
import torch

from oracle import muse_oracle as orc
from tests.gpu_util import Case, kernels_launched, rel_err, to_dev, to_np, tol
from tests.test_gpu_cluster import CASES
from tests.test_gpu_forward import TC_BWD_KERNELS, TC_FWD_KERNELS, _forward_parity

pytestmark = pytest.mark.gpu

# 32 planes (the last that fit) and several key chunks a cluster; 33 planes; a second tile of query clusters; 79 planes
MANY = [("d64", 20, 9, 3, 33), ("d64", 50, 40, 4, 34), ("d128", 130, 24, 4, 40), ("d64", 12, 10, 2, 80), ("d128", 16, 40, 5, 80)]


@pytest.mark.parametrize("base,Cq,Ck,m,S", MANY)
def test_forward_and_backward_of_many_blocks(base, Cq, Ck, m, S):
    """The backward with output gradients in the late blocks alone (from block 33 on, where there are as many): the gradients of the
    keys before them then come through the last planes and nothing else, so a plane that is lost shows."""
    from paper_2509_10406_b200 import binding as mb
    w = CASES[base].with_(Hq=2, Hkv=1, N=62 * S, S=S, Cq=Cq, Ck=Ck, m=m, components=64)
    _forward_parity(w, 128.0, expect_kernels=TC_FWD_KERNELS)
    c = Case(w)
    late = min(33, S - 1) * (w.N // S)
    c.dO[:, :, :late] = 0
    qbar32 = c.qbar.astype(np.float32)
    p = c.params()
    buf = mb.MuseBuffers(p, backward=True)
    Q, K, V, dO = c.dev()
    aq, qb = to_dev(c.a_q, "i"), to_dev(qbar32, "f32")
    with kernels_launched() as rec:
        mb.muse_summarize(p, K, V, to_dev(c.a_k, "i"), qb, buf.off_k, buf.perm_k, buf.summaries, buf.ws)
        mb.muse_attn_fwd(p, Q, K, V, aq, qb, buf.off_k, buf.perm_k, buf.summaries, None, buf.O, buf.LSE, buf.sel, buf.ws)
        mb.muse_attn_bwd(p, Q, K, V, buf.O, buf.LSE, dO, aq, qb, buf.off_k, buf.perm_k, buf.summaries, buf.sel, buf.dQ, buf.dK, buf.dV, buf.ws)
        torch.cuda.synchronize()
    assert mb.muse_status(buf.ws) == 0 and TC_BWD_KERNELS <= rec.names, sorted(rec.names)
    e = orc.layer_backward(*(x.astype(np.float64) for x in (c.Q, c.K, c.V, c.dO)), c.a_q, c.a_k, qbar32.astype(np.float64),
                           sigma=c.sigma, S=S, Ck=Ck, m=m, causal=True, sel=to_np(buf.sel)[..., :m], sel_mode=0, agg_grad=True)
    errs = dict(dQ=rel_err(to_np(buf.dQ), e[0]), dK=rel_err(to_np(buf.dK)[:, :, :late], e[1][:, :, :late]),
                dV=rel_err(to_np(buf.dV)[:, :, :late], e[2][:, :, :late]))
    print(base, S, errs)
    assert all(v <= tol(w.dtype) for v in errs.values()), errs


@pytest.mark.parametrize("base,N,Ck,m,S", [("d64", 8192, 1024, 4, 32), ("d64", 8192, 4096, 8, 8)])
def test_retrieval_index_with_the_most_buckets(base, N, Ck, m, S):
    """One head whose index takes the largest thread-block cluster (16 CTAs where the device holds them) at 124 and 112 KB a CTA."""
    w = CASES[base].with_(Hq=1, Hkv=1, N=N, S=S, Cq=4, Ck=Ck, m=m, components=64)
    _forward_parity(w, 128.0, expect_kernels={"k_ret_index"})
