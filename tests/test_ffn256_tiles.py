"""The d = 256 FFN kernel (fe_ffn256.cu) with several tiles per CTA: the next
tile's A lands k block by k block while the previous tile's stores drain.  More
rows than 128 per SM for the element layers (with and without a Q tail) and the
SeqEnc block, the last tile partial, against the oracle."""
import numpy as np
import pytest

import oracle.fe_oracle as O
from oracle import compare
from paper_2603_02565_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_02565_gb300 import build
    build.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("kw", [dict(B=97, K=401, M=451, Ly=1), dict(B=71, K=501, M=301, Ly=3),
                                dict(B=201, K=301, M=251, Ly=2)], ids=lambda k: "B%(B)d_K%(K)d_M%(M)d_Ly%(Ly)d" % k)
def test_tiles(dev, kw):
    from paper_2603_02565_gb300.binding import Evaluator
    w = wl.stress(C=64, L=3, **kw)
    ev = Evaluator(w.cfg, w.weights)
    ctx, pool = (torch.from_numpy(a).to(dev, torch.bfloat16) for a in (w.context, w.pool))
    s, b = ev.evaluate(ctx, pool, torch.from_numpy(w.cand_idx).to(dev))
    ev.close()
    s, b = s.cpu().numpy(), b.cpu().numpy()
    rq = [0, kw["B"] // 2, kw["B"] - 1]
    o_s, o_b, _, _ = O.evaluate(w.context, w.pool, w.cand_idx, w.weights, w.cfg, requests=rq)
    # relative to the request's largest score: a score is a sum of signed terms, and among a request's
    # hundreds some cancel to a fraction of the terms their rounding is relative to
    err = np.abs(s[rq] - o_s[rq]).max(axis=1) / np.abs(o_s[rq]).max(axis=1)
    assert (err <= compare.REL_TOL).all(), err
    assert compare.best_ok(b[rq], o_s[rq], o_b[rq])[0]
