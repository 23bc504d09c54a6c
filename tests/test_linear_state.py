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


# keys around `mean` in every row of the context, or in every seventh feature only
NEGATIVE = [(-9.0, 1, 300, 64, 2), (-15.0, 1, 65, 64, 1), (-20.0, 1, 500, 64, 2), (-20.0, 7, 500, 128, 4),
            (-40.0, 1, 1100, 32, 1), (-60.0, 1, 130, 256, 8)]


@pytest.mark.parametrize("mean,every,C,d,H", NEGATIVE)
def test_strongly_negative_keys(dev, mean, every, C, d, H):
    """phi(K) = exp(K) far below f16's smallest number: an attended value is a ratio of sums
    of it, finite and as exact as the keys.  Every context row is +-1 plus noise (its
    LayerNorm the same direction), which W_K turns into keys around `mean`."""
    from paper_2603_02565_gb300.binding import Evaluator
    w = wl.make_workload("serving", B=3, M=40, C=C, d=d, H=H, Ly=1, K=4, L=3, linear_context_attn=True, encode_pool=True)
    rng = np.random.default_rng(5)
    bf16 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).bfloat16().float().numpy()
    u = np.where(np.arange(d) % 2 == 0, 1.0, -1.0)
    context = bf16(u + 0.05 * rng.standard_normal((3, C, d)))
    weights = dict(w.weights)
    wk = 0.3 * rng.standard_normal((d, d))
    wk -= np.outer(u, u @ wk) / d  # the noise alone spreads the keys
    wk[:, ::every] += mean / d * u[:, None]
    weights["WK.0"] = bf16(wk)
    weights["WV.0"] = bf16(rng.standard_normal((d, d)))
    weights["WO.0"] = bf16(0.2 * rng.standard_normal((d, d)))
    ev = Evaluator(w.cfg, weights)
    ctx, pool = (torch.from_numpy(a).to(dev, torch.bfloat16) for a in (context, w.pool))
    ev.evaluate(ctx, pool, torch.from_numpy(w.cand_idx).to(dev))
    elem = ev.fetch("elem").reshape(3, 40, d)
    ev.close()
    for b in range(3):
        kv = O.context_kv(context[b].astype(np.float64), weights, 1, w.cfg.ln_eps)
        assert kv[0][0][:, ::every].mean() == pytest.approx(mean, rel=0.02)
        ref = O.encode_elements(w.pool[b].astype(np.float64), kv, weights, H, w.cfg.ln_eps, linear=True)
        # a key around -60 is rounded by up to 2^-6 in f16, so phi by 2^-6 of itself; independent over the rows
        np.testing.assert_allclose(elem[b], ref, rtol=1e-3, atol=2e-3 + 2.0 ** -10 * abs(mean) / C ** 0.5)
