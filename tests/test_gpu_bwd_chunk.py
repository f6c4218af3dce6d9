"""The backward over chunks (csrc/lmhead_bwd_chunk.cu) where its tile list can go
wrong: one row, tiles and chunks with remainders in both directions, a last H
tile of 64 to 192 columns, one and several token chunks (dW stored or added to),
buffers used again, the entropy term, a call without any gradient row, and the lines
of the rule that chooses it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2607_21653_gb300 as molt  # noqa: E402
from oracle import molt_oracle as O  # noqa: E402
from workloads import random_problem  # noqa: E402

from parity import assert_grad_close, assert_loss_close, behavior_from_oracle, bf, np_, t  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    molt.build()
    molt.load()


def _run(args, **kw):
    out = molt.policy_loss_fwd_bwd_ex(*args, 0.2, 0.28, **kw)
    torch.cuda.synchronize()
    assert molt.device_status() == 0
    return out


# (1, 640, 1): one row, one column; (257, 704, 513): remainders of one row, column
# and a 192-column H tile; (512, 320, 4097): the rule's least T for this H, a
# 64-column H tile; (300, 256, 4096), (700, 256, 20481), (769, 256, 8200): its lines at
# H = 256; (1500, 256, 10000): chunks of 8 x 4 tiles, ten of the vocabulary; (2049, 640,
# 2100): of 8 x 8, two of the vocabulary (the rows with a gradient are fewer than 2048);
# (4200, 1088, 4400): two of tokens and three of the vocabulary, a 64-column H tile.
# None of them has more chunks than buffers: see test_buffers_used_again
@pytest.mark.parametrize("T,H,V", [(1, 640, 1), (257, 704, 513), (512, 320, 4097), (300, 256, 4096), (700, 256, 20481),
                                   (769, 256, 8200), (1500, 256, 10000), (2049, 640, 2100), (4200, 1088, 4400)])
def test_chunk_backward_matches_oracle(T, H, V):
    rng = np.random.default_rng(T + H + V)
    h, W, x, m = random_problem(rng, T, H, V, mask_frac=0.1 if T > 1 else 0.0, w_std=0.05)
    m[-1] = 1
    adv = rng.standard_normal(T).astype(np.float32)
    h64, W64 = O.widen_bf16(h), O.widen_bf16(W)
    b = behavior_from_oracle(h64, W64, x, 0.3, 0.2, 0.28, T)
    ref = O.policy_loss(h64, W64, x, b.astype(np.float64), adv.astype(np.float64), m, 0.2, 0.28)
    ref["_adv"] = adv.astype(np.float64)
    args = (bf(h), bf(W), t(x), t(b), t(adv), t(m))
    out = _run(args)
    assert_loss_close(float(out["loss"].item()), ref)
    assert_grad_close(np_(out["dhidden"]), ref["dH"], "dhidden")
    assert_grad_close(np_(out["dW"]), ref["dW"], "dW")
    # added onto the caller's dW instead of stored
    dW0 = torch.randn(V, H, device="cuda", generator=torch.Generator(device="cuda").manual_seed(T))
    acc = dW0.clone()
    _run(args, dW=acc, accumulate_dW=True)
    assert_grad_close(np_(acc - dW0), ref["dW"], "dW accumulated")
    # the entropy term's gradient is linear in its coefficient (against the oracle:
    # test_entropy_term_alone)
    e1, e2 = (_run(args, entropy_coef=c) for c in (0.01, 0.02))
    d1, d2 = (np_(e["dW"]) - np_(out["dW"]) for e in (e1, e2))
    if V > 1:
        assert np.abs(d2 - 2 * d1).max() <= 2e-2 * np.abs(d2).max() + 2e-2 * np.abs(ref["dW"]).max()
    # no row with a gradient: everything 0, dW included, whatever it held
    dW = torch.full((V, H), float("nan"), device="cuda")
    zero = _run((*args[:4], torch.zeros_like(args[4]), args[5]), dW=dW)
    assert (np_(zero["dW"]) == 0).all() and (np_(zero["dhidden"]) == 0).all()
    if H % 128 == 0:
        det = [_run(args, deterministic=True, det_clusters=n) for n in (0, 0, 4)]
        assert_grad_close(np_(det[0]["dW"]), ref["dW"], "dW deterministic")
        for o in det[1:]:
            for k in ("dW", "dhidden"):
                np.testing.assert_array_equal(np_(o[k]).view(np.uint8), np_(det[0][k]).view(np.uint8), err_msg=k)


def _all_live(T, H, V, w_std):
    """A problem whose every row has a gradient: nothing masked, ratios inside the clip band."""
    rng = np.random.default_rng(T + 3 * H + V)
    h, W, x, m = random_problem(rng, T, H, V, mask_frac=0.0, w_std=w_std)
    m[:] = 1
    h64, W64 = O.widen_bf16(h), O.widen_bf16(W)
    b = behavior_from_oracle(h64, W64, x, 0.02, 0.2, 0.28, T)
    return rng, h, W, x, m, b, h64, W64


# each kind of ring with at least twice as many chunks as buffers, so that every buffer
# is written again after its readers: 8 x 4 tiles in sixteen buffers, two chunks of tokens;
# 4 x 8 in sixteen; 8 x 8 in eight, two chunks of tokens, a 192-column H tile; 16 x 16 in
# two, two chunks of tokens, a 64-column H tile
@pytest.mark.parametrize("T,H,V", [(2305, 256, 17000), (520, 320, 66000), (2100, 704, 14700), (4300, 2112, 8300)])
def test_buffers_used_again(T, H, V):
    plan = molt.backward_plan(T, H, V)
    tiles = lambda n, chunk: -(-(-(-n // 256)) // (chunk // 256))
    assert plan["kernel"] == "lmhead_bwd_chunk_kernel"
    assert tiles(T, plan["chunk_tokens"]) * tiles(V, plan["chunk_columns"]) >= 2 * plan["buffers"]
    rng, h, W, x, m, b, h64, W64 = _all_live(T, H, V, 0.05)
    adv = (np.sign(rng.standard_normal(T)) * rng.uniform(0.5, 2.0, T)).astype(np.float32)
    ref = O.policy_loss(h64, W64, x, b.astype(np.float64), adv.astype(np.float64), m, 0.2, 0.28)
    ref["_adv"] = adv.astype(np.float64)
    args = (bf(h), bf(W), t(x), t(b), t(adv), t(m))
    dW0 = torch.randn(V, H, device="cuda", generator=torch.Generator(device="cuda").manual_seed(T))
    runs = [dict(), dict(dW=dW0.clone(), accumulate_dW=True)] + [dict(deterministic=True)] * (H % 128 == 0)
    for kw in runs:
        out = _run(args, **kw)
        assert molt.stats_dict(out["stats"])["n_grad_rows"] == T
        assert_loss_close(float(out["loss"].item()), ref)
        assert_grad_close(np_(out["dhidden"]), ref["dH"], "dhidden")
        dW = out["dW"] - dW0 if "dW" in kw else out["dW"]
        assert_grad_close(np_(dW), ref["dW"], "dW")


# A = 0: the entropy term is the whole gradient
@pytest.mark.parametrize("T,H,V", [(1, 640, 7), (257, 704, 513), (512, 320, 4097), (300, 256, 4096), (4200, 1088, 4400),
                                   (2305, 256, 17000)])
def test_entropy_term_alone(T, H, V):
    assert molt.backward_plan(T, H, V)["kernel"] == "lmhead_bwd_chunk_kernel"
    _, h, W, x, m, b, h64, W64 = _all_live(T, H, V, 3.2 / H ** 0.5)
    adv = np.zeros(T, np.float32)
    ref = O.policy_loss_ex(h64, W64, x, b.astype(np.float64), adv.astype(np.float64), m, 0.2, 0.28, entropy_coef=0.1)
    out = _run((bf(h), bf(W), t(x), t(b), t(adv), t(m)), entropy_coef=0.1)
    assert molt.stats_dict(out["stats"])["n_grad_rows"] == T
    assert_grad_close(np_(out["dhidden"]), ref["dH"], "dhidden")
    assert_grad_close(np_(out["dW"]), ref["dW"], "dW")
