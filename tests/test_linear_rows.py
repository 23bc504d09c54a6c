"""The linear-attention rows kernel (fe_linattn.cu, lin_attn_kernel): segments
whose rows are dealt out to one, two, four and eight CTAs, more rows than the
CTAs take in one turn, a single row, and the widest states, against the oracle."""
import numpy as np
import pytest

import oracle.fe_oracle as O
from oracle import compare
from paper_2603_02565_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (B, K, L, M, d, heads)
CASES = [(609, 30, 5, 90, 64, 2), (300, 40, 4, 75, 64, 1), (200, 50, 4, 70, 128, 4), (140, 60, 4, 80, 64, 2),
         (3, 300, 5, 400, 64, 2), (2, 1, 1, 1, 128, 2), (610, 20, 3, 40, 512, 8), (5, 90, 4, 150, 256, 8)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_02565_gb300 import build
    build.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("case", CASES, ids=lambda c: "B%d_K%d_L%d_M%d_d%d_h%d" % c)
def test_rows(dev, case):
    from paper_2603_02565_gb300.binding import Evaluator
    B, K, L, M, d, H = case
    w = wl.make_workload("serving", B=B, K=K, L=L, M=M, C=24, d=d, H=H, Ly=1, linear_context_attn=True)
    ev = Evaluator(w.cfg, w.weights)
    ctx, pool = (torch.from_numpy(a).to(dev, torch.bfloat16) for a in (w.context, w.pool))
    s, b = ev.evaluate(ctx, pool, torch.from_numpy(w.cand_idx).to(dev))
    ev.close()
    s, b = s.cpu().numpy(), b.cpu().numpy()
    rq = [0, B - 1]
    o_s, o_b, _, _ = O.evaluate(w.context, w.pool, w.cand_idx, w.weights, w.cfg, requests=rq)
    # relative to the request's largest score: a score is a sum of d signed terms, and some cancel to a
    # fraction of the terms their rounding is relative to
    err = np.abs(s[rq] - o_s[rq]).max(axis=1) / np.abs(o_s[rq]).max(axis=1)
    assert (err <= compare.REL_TOL).all(), err
    assert compare.best_ok(b[rq], o_s[rq], o_b[rq])[0]
