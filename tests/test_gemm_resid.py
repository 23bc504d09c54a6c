"""The residual rows of the LayerNorm GEMMs (fe_gemm.cu), which a warp loads
into its own staging buffers: every width up to 128 columns (at d = 32 half of
the warps have no block), one tile per CTA and several, the last one partial,
split weights (fp32 models), the clusters of 128 and of 64 columns per CTA, and
rows wider than 128 columns on one CTA, against the oracle."""
import numpy as np
import pytest

import oracle.fe_oracle as O
from oracle import compare
from paper_2603_02565_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (B, K, d, heads, fp32): K > 128 keeps the sequence side on the GEMM kernels
CASES = [(2, 131, 32, 1, False), (301, 140, 32, 1, False), (3, 200, 64, 2, True), (151, 301, 64, 1, False),
         (5, 129, 128, 4, True), (97, 401, 128, 4, False), (3, 130, 256, 8, True), (150, 131, 256, 4, False),
         (2, 140, 512, 8, False), (40, 257, 512, 8, False), (160, 140, 512, 16, False)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_02565_gb300 import build
    build.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("case", CASES, ids=lambda c: "B%d_K%d_d%d_h%d_fp32%d" % c)
def test_residual_rows(dev, case):
    from paper_2603_02565_gb300.binding import Evaluator
    B, K, d, H, fp32 = case
    w = wl.make_workload("serving", B=B, K=K, L=3, M=30, C=16, d=d, H=H, Ly=1, io_bf16=not fp32)
    ev = Evaluator(w.cfg, w.weights)
    dt = torch.float32 if fp32 else torch.bfloat16
    ctx, pool = (torch.from_numpy(a).to(dev, dt) for a in (w.context, w.pool))
    s, b = ev.evaluate(ctx, pool, torch.from_numpy(w.cand_idx).to(dev))
    ev.close()
    s, b = s.cpu().numpy(), b.cpu().numpy()
    rq = [0, B - 1]
    o_s, o_b, _, _ = O.evaluate(w.context, w.pool, w.cand_idx, w.weights, w.cfg, requests=rq)
    # relative to the request's largest score: a score is a sum of d signed terms, and among a request's
    # hundreds some cancel to a fraction of the terms their rounding is relative to
    err = np.abs(s[rq] - o_s[rq]).max(axis=1) / np.abs(o_s[rq]).max(axis=1)
    assert (err <= compare.REL_TOL).all(), err
    assert compare.best_ok(b[rq], o_s[rq], o_b[rq])[0]
