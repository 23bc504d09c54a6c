"""The [CLS] attention for many sequences (fe_misc.cu, cls_rows_kernel: 32 / heads
sequences per warp) against the oracle's scores: each width and head size it is
built for, sequence counts that leave a partial last warp, L at its smallest and
at the staged and unstaged sizes of the position table, and a rejected request
between valid ones."""
import numpy as np
import pytest

import oracle.fe_oracle as O
from oracle import compare
from paper_2603_02565_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (B, K, L, d, heads): at least 4000 warps of 32 / heads sequences
CASES = [(161, 401, 3, 64, 2), (257, 500, 1, 64, 1), (17, 1901, 10, 128, 4), (65, 1000, 32, 128, 2),
         (5, 3301, 10, 256, 8), (13, 2501, 25, 256, 4), (3, 2671, 13, 512, 16), (4, 4096, 5, 512, 8)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_02565_gb300 import build
    build.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("case", CASES, ids=lambda c: "B%d_K%d_L%d_d%d_h%d" % c)
def test_many_sequences(dev, case):
    from paper_2603_02565_gb300.binding import FE_ERR_INDEX, Evaluator
    B, K, L, d, H = case
    w = wl.make_workload("serving", B=B, K=K, L=L, M=40, C=32, d=d, H=H, Ly=1)
    w.cand_idx[1, K // 2, 0] = 40  # request 1 is rejected
    ev = Evaluator(w.cfg, w.weights)
    ctx, pool = (torch.from_numpy(a).to(dev, torch.bfloat16) for a in (w.context, w.pool))
    s, b = ev.evaluate(ctx, pool, torch.from_numpy(w.cand_idx).to(dev))
    assert ev.last_status == FE_ERR_INDEX
    ev.close()
    s, b = s.cpu().numpy(), b.cpu().numpy()
    assert np.isnan(s[1]).all() and b[1] == -1
    rq = [0, B - 1]
    o_s, o_b, _, _ = O.evaluate(w.context, w.pool, w.cand_idx, w.weights, w.cfg, requests=rq)
    # a score is a sum of d signed terms, and its rounding error is relative to the terms: among the thousands of
    # scores of a request a few cancel to a fraction of them, so the bound is relative to the request's largest score
    err = np.abs(s[rq] - o_s[rq]).max(axis=1) / np.abs(o_s[rq]).max(axis=1)
    assert (err <= compare.REL_TOL).all(), err
    assert compare.best_ok(b[rq], o_s[rq], o_b[rq])[0]
