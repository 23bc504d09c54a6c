"""The attention kernel (fe_attn.cu) inside whole batches, against the oracle's scores:
element -> context attention over fixed-length contexts (Section 4.2) and the
cross-sequence attention over K sequences (Section 4.4) whose last key chunk is
partial (K = 1000 and K = 200 are not multiples of 64: V rows past the key count are
zeroed).  The stress batch of 24 requests gives a group of warps several units, some
of them query tiles past their request's distinct elements (skipped).  The wide
cross-sequence batch has three query tiles per request and more (request, head) pairs
than the groups of one round."""
import numpy as np
import pytest

import oracle.fe_oracle as O
from oracle import compare
from paper_2603_02565_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# name: (workload, its sizes, requests checked (None: all))
CASES = {"serving": ("serving", dict(B=4), None),
         "ksweep_K1000": ("ksweep", dict(B=2, K=1000), None),
         "stress": ("stress", dict(B=3), None),
         "stress24": ("stress", dict(B=24), [0, 11, 23]),
         "cross_three_tiles": ("serving", dict(B=160, K=300, M=40, C=64), [0, 77, 151, 159])}


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_02565_gb300 import build
    build.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("case", sorted(CASES))
def test_attention_in_a_batch(dev, case):
    from paper_2603_02565_gb300.binding import Evaluator
    kind, sizes, rq = CASES[case]
    w = wl.make_workload(kind, **sizes)
    rq = list(range(sizes["B"])) if rq is None else rq
    ev = Evaluator(w.cfg, w.weights)
    dt = torch.bfloat16 if w.cfg.io_bf16 else torch.float32
    ctx, pool = (torch.from_numpy(a).to(dev, dt) for a in (w.context, w.pool))
    s, b = ev.evaluate(ctx, pool, torch.from_numpy(np.ascontiguousarray(w.cand_idx)).to(dev))
    s, b = s.cpu().numpy(), b.cpu().numpy()
    ev.close()
    o_s, o_b, _, _ = O.evaluate(w.context, w.pool, w.cand_idx, w.weights, w.cfg, requests=rq)
    err = compare.score_error(s[rq], o_s[rq])
    ok, _ = compare.best_ok(b[rq], o_s[rq], o_b[rq])
    assert err <= compare.REL_TOL, f"max rel err {err:.3e}"
    assert ok
