"""Work distribution of the attention kernel (fe_attn.cu): rounds over blocks of
segments and query tiles.  Elements encoded over the whole pool make every
request span ceil(M / 128) query tiles with a partial last one; the shapes take
one, two and three tiles, more segments than one round holds, several tiles per
round (few segments), both head sizes, and row counts at the edges of a tile and of
a 32-row block.  The element encodings of sampled requests are compared with the
oracle (f16 attention operands, 2^-11 relative each, over rows of unit variance)."""
import numpy as np
import pytest

import oracle.fe_oracle as O
from paper_2603_02565_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (B, M, C, d, heads): requests, pool rows (= query rows), keys, width, heads of 32 or 64 columns
CASES = [(3, 1, 64, 64, 2), (40, 300, 70, 128, 4), (200, 129, 65, 128, 4), (2, 385, 1, 128, 4), (160, 33, 128, 64, 2),
         (60, 257, 130, 128, 2), (170, 96, 129, 64, 1), (5, 128, 300, 128, 2)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_02565_gb300 import build
    build.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("case", CASES, ids=lambda c: "B%d_M%d_C%d_d%d_h%d" % c)
def test_query_tiles_and_segments(dev, case):
    from paper_2603_02565_gb300.binding import Evaluator
    B, M, C, d, H = case
    w = wl.make_workload("serving", B=B, M=M, C=C, d=d, H=H, K=4, L=1, encode_pool=True)
    ev = Evaluator(w.cfg, w.weights)
    ctx, pool = (torch.from_numpy(a).to(dev, torch.bfloat16) for a in (w.context, w.pool))
    ev.evaluate(ctx, pool, torch.from_numpy(w.cand_idx).to(dev))
    elem = ev.fetch("elem").reshape(B, M, d)
    ev.close()
    for b in sorted({0, B // 2, B - 1}):
        kv = O.context_kv(w.context[b], w.weights, w.cfg.n_layers, w.cfg.ln_eps)
        ref = O.encode_elements(w.pool[b].astype(np.float64), kv, w.weights, H, w.cfg.ln_eps)
        np.testing.assert_allclose(elem[b], ref, rtol=1e-3, atol=2e-3)
