"""Masked vocabularies (constrained decoding) on every epilogue of the round:
base logits masked with the type's lowest value or with -inf, and NaN among
-inf, against float64 log-softmax.

The head is zero, so each stage's logits are its base logits and the reference
needs no matrix (the widest head would take gigabytes in 64 bits).  Every
parent of a depth then has the same children, and a node's score is the sum of
its path's log-softmax values; the tolerance is the round's own (1e-4 on
cumulative log-probabilities).
"""
import numpy as np
import pytest
import torch

from tests.gpu_util import LOGP_TOL

pytestmark = pytest.mark.gpu

LOWEST = np.finfo(np.float32).min

# one shape per epilogue, with several tiles to a slot where it has tiles
SHAPES = {
    # a warp to a row: up to 16 rows, up to 32 with long lists; heads that
    # stay in L2 and heads above three times L2 (walked backwards in odd stages)
    "rows8": dict(V=81000, H=64, k=8, batch=1),
    "rows1": dict(V=81000, H=64, k=1, batch=1),
    "rows24_k12": dict(V=81000, H=64, k=12, batch=2),
    "rows8_streamed": dict(V=160001, H=1400, k=8, batch=1),
    "rows32_k16_streamed": dict(V=160001, H=1400, k=16, batch=2),
    # a thread to a row
    "rows128": dict(V=81000, H=64, k=8, batch=16),
    "rows64_k32": dict(V=81000, H=64, k=32, batch=2),
    "rows128_streamed": dict(V=160001, H=1400, k=8, batch=16),
    # CTA pairs
    "rows256_pairs": dict(V=81000, H=64, k=16, batch=16),
    # the fused round (set by the stall hook), 8-row and 16-row instances
    "fused_rows8": dict(V=81000, H=64, k=8, batch=1, fused=True),
    "fused_rows16": dict(V=81000, H=64, k=8, batch=2, fused=True),
    # f32 heads: fine and whole chunks of the partials pass
    "f32_rows4": dict(V=40000, H=8, k=4, batch=1, dtype="f32"),
    "f32_rows136": dict(V=40000, H=8, k=8, batch=17, dtype="f32"),
}
DEPTHS = 3


def allowed_columns(V, pattern):
    """Columns left unmasked per depth [DEPTHS][V]: a sparse allow-list, or a
    vocabulary whose head or tail is masked (the first columns that a forward
    or a backward walk meets)."""
    keep = np.zeros((DEPTHS, V), bool)
    for d in range(DEPTHS):
        if pattern == "sparse":
            keep[d, np.random.default_rng(d).choice(V, 400, replace=False)] = True
        elif pattern == "head_masked":
            keep[d, V - V // 3 - d:] = True
        else:
            keep[d, :V // 3 + d] = True
    return keep


def draft(shape, L, nan_row=None):
    from paper_2608_02123_gb300 import pctree as P
    s = dict(shape)
    fused, dtype = s.pop("fused", False), s.pop("dtype", "bf16")
    cfg = P.make_config(s["V"], s["H"], DEPTHS, s["k"], 40, s["batch"], weight_dtype=dtype)
    W = torch.zeros(s["V"], s["H"], device="cuda",
                    dtype=torch.bfloat16 if dtype == "bf16" else torch.float32)
    if nan_row is not None:
        W[nan_row] = float("nan")
    root = torch.zeros(s["batch"], dtype=torch.int32, device="cuda")
    dr = P.Drafter(cfg, with_pool=True)
    if fused:
        P.pctree_debug_stall_stage(1 << 20, 1_000_000_000)
    try:
        return dr.draft(torch.from_numpy(L).cuda(), W, W, root).to_host()
    finally:
        P.pctree_debug_stall_stage(-1, 1_000_000_000)


def check_pool(host, L, k):
    """Children and scores of every parent of every request."""
    assert int(host["status"][0]) == 0
    for r in range(L.shape[0]):
        tok, par, logp = (host[n][r] for n in ("pool_token", "pool_parent", "pool_logp"))
        base = 1
        for d in range(DEPTHS):
            z = L[r, d].astype(np.float64)
            best = np.argsort(-z, kind="stable")[:k]
            m = z.max()
            step = z[best] - (m + np.log(np.exp(z - m).sum()))
            for _ in range(1 if d == 0 else k):
                np.testing.assert_array_equal(tok[base:base + k], best)
                np.testing.assert_allclose(logp[base:base + k], logp[par[base]] + step,
                                           rtol=0, atol=LOGP_TOL)
                base += k


@pytest.mark.parametrize("pattern", ["sparse", "head_masked", "tail_masked"])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_lowest_value_masks(name, pattern):
    """A mask of the lowest finite float leaves probability 0 and changes
    neither the status nor the other children's scores."""
    s = SHAPES[name]
    keep = allowed_columns(s["V"], pattern)
    rng = np.random.default_rng(41)
    L = rng.normal(0.0, 4.0, (s["batch"], DEPTHS, s["V"])).astype(np.float32)
    L[:, ~keep] = LOWEST
    check_pool(draft(s, L), L, s["k"])


@pytest.mark.parametrize("name", sorted(SHAPES))
def test_wholly_masked_rows(name):
    """Rows that hold nothing but the lowest value are uniform."""
    s = SHAPES[name]
    L = np.full((s["batch"], DEPTHS, s["V"]), LOWEST, np.float32)
    check_pool(draft(s, L), L, s["k"])


@pytest.mark.parametrize("where", ["logits", "weights"])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_nan_among_neg_inf(name, where):
    """A NaN base logit, or one that a NaN weight makes, is reported also where
    every other logit near it is -inf (which is legal), and the finite
    logits are still the row's first children."""
    s = SHAPES[name]
    V, k = s["V"], s["k"]
    L = np.full((s["batch"], DEPTHS, V), -np.inf, np.float32)
    cols = V // 2 + np.arange(k)
    L[:, :, cols] = np.linspace(5.0, 3.0, k, dtype=np.float32)
    assert int(draft(s, L)["status"][0]) == 0
    at = V // 5 + 3
    nan_row = None
    if where == "logits":
        L[-1, 0, at] = np.nan
    else:
        nan_row = at
    host = draft(s, L, nan_row)
    assert int(host["status"][0]) == -5                # PCTREE_ERR_NONFINITE
    np.testing.assert_array_equal(host["pool_token"][-1][1:1 + k], cols)
