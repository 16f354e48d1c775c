"""GPU: the rows that a tile of retrieved keys brings beside the keys its queries see (later blocks of the cluster, the next cluster,
the next head) never reach a result, whatever they hold."""
import numpy as np
import pytest
import torch

from tests.gpu_util import Case, rel_err, to_dev, to_np
from tests.test_gpu_cluster import CASES

pytestmark = pytest.mark.gpu


# keys per cluster on both sides of the rules that choose the forward and backward kernels; the last two retrieve blocks (buckets)
@pytest.mark.parametrize("base,Ck,m,k2", [("d64", 7, 3, 0), ("d64", 13, 3, 0), ("d64", 20, 11, 0), ("d64", 40, 5, 0), ("d128", 9, 3, 0),
                                          ("d128", 25, 4, 0), ("d128", 40, 5, 0), ("d64", 7, 3, 1), ("d128", 9, 3, 2)])
def test_keys_that_nobody_sees_may_hold_anything(base, Ck, m, k2):
    from paper_2509_10406_b200 import binding as mb
    S, N = 4, 2040
    w = CASES[base].with_(Hq=4, Hkv=2, N=N, S=S, Cq=9, Ck=Ck, m=m, components=64)
    c = Case(w, gain=128.0)
    p = c.params(k2=k2)
    buf = mb.MuseBuffers(p, backward=True)
    Q, K, V, dO = c.dev()
    aq, qb = to_dev(c.a_q, "i"), to_dev(c.qbar.astype(np.float32), "f32")
    mb.muse_summarize(p, K, V, to_dev(c.a_k, "i"), qb, buf.off_k, buf.perm_k, buf.summaries, buf.ws)

    def both():
        mb.muse_attn_fwd(p, Q, K, V, aq, qb, buf.off_k, buf.perm_k, buf.summaries, None, buf.O, buf.LSE, buf.sel, buf.ws, bsel_out=buf.bsel)
        assert mb.muse_status(buf.ws) == 0
        mb.muse_attn_bwd(p, Q, K, V, buf.O, buf.LSE, dO, aq, qb, buf.off_k, buf.perm_k, buf.summaries, buf.sel, buf.dQ, buf.dK, buf.dV,
                         buf.ws, bsel=buf.bsel)
        assert mb.muse_status(buf.ws) == 0
        return [to_np(x) for x in (buf.O, buf.LSE, buf.dQ, buf.dK, buf.dV)]

    clean = both()
    # the bucketed keys and values that retrieval reads: NaN in the last block (no query retrieves it) and in all of the second kv head
    lay = mb.muse_summaries_layout(p)
    last = np.nonzero(to_np(buf.perm_k)[0, 0] // (N // S) == S - 1)[0]
    assert last.size == N // S
    for off in lay[5:7]:
        rows = buf.summaries[off:off + 2 * N * w.D * 2].view(torch.bfloat16).view(2, N, w.D)
        rows[0, torch.from_numpy(last).cuda()] = float("nan")
        rows[1] = float("nan")
    O, L, dQ, dK, dV = both()
    assert np.array_equal(O[:, :2], clean[0][:, :2]) and np.array_equal(L[:, :2], clean[1][:, :2])
    assert np.array_equal(dQ[:, :2], clean[2][:, :2])
    # (dK and dV are sums in no fixed order, rounded to bf16 once)
    assert rel_err(dK[:, 0], clean[3][:, 0]) <= 8e-3 and rel_err(dV[:, 0], clean[4][:, 0]) <= 8e-3
