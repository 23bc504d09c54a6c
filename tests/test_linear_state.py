"""The context-state kernel of the linear-attention module (fe_linattn.cu) at the
edges of its 64-row chunks and for each feature-group width (32, 64 and 128 columns,
heads of 32 and 64): the element encodings, which read the states, against the
oracle.  One layer or three keep the fused state mode of the context kernel out."""
import numpy as np
import pytest

import oracle.fe_oracle as O
from paper_2603_02565_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (rows C, d, heads, layers)
CASES = [(1, 64, 2, 1), (63, 64, 1, 1), (64, 128, 4, 1), (65, 128, 2, 3), (128, 64, 2, 3), (129, 32, 1, 1),
         (500, 256, 8, 1)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_02565_gb300 import build
    build.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("case", CASES, ids=lambda c: "C%d_d%d_h%d_l%d" % c)
def test_context_states(dev, case):
    from paper_2603_02565_gb300.binding import Evaluator
    C, d, H, Ly = case
    w = wl.make_workload("serving", B=5, M=40, C=C, d=d, H=H, Ly=Ly, K=4, L=3, linear_context_attn=True,
                         encode_pool=True)
    ev = Evaluator(w.cfg, w.weights)
    ctx, pool = (torch.from_numpy(a).to(dev, torch.bfloat16) for a in (w.context, w.pool))
    ev.evaluate(ctx, pool, torch.from_numpy(w.cand_idx).to(dev))
    elem = ev.fetch("elem").reshape(5, 40, d)
    ev.close()
    for b in range(5):
        kv = O.context_kv(w.context[b], w.weights, Ly, w.cfg.ln_eps)
        ref = O.encode_elements(w.pool[b].astype(np.float64), kv, w.weights, H, w.cfg.ln_eps, linear=True)
        # f16 keys, values and queries: 2^-11 relative each, two layers' worth of rows of unit variance
        np.testing.assert_allclose(elem[b], ref, rtol=1e-3, atol=2e-3)
