"""The forward on CTA pairs and the merge of its partials where they can go wrong:
one row and one column, an empty second half of a tile (rows or vocab columns),
remainders around 128 and 256 in both, more than one group of 16 token tiles, one
K block, and a few rows against many vocab splits (hundreds of partials a row)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2607_21653_gb300 as molt  # noqa: E402
from oracle import molt_oracle as O  # noqa: E402
from workloads import random_problem  # noqa: E402

from parity import LOGP_ATOL, bf, np_, t  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    molt.build()
    molt.load()


@pytest.mark.parametrize("T,H,V", [(1, 64, 1), (128, 128, 128), (129, 64, 129), (257, 192, 385), (300, 320, 1000),
                                   (4353, 128, 700), (40, 256, 40001)])
@pytest.mark.parametrize("call", ["token_logprobs", "token_logprobs_noalloc"])
def test_forward_matches_oracle(T, H, V, call):
    rng = np.random.default_rng(T + H + V)
    h, W, x, m = random_problem(rng, T, H, V, mask_frac=0.3 if T > 1 else 0.0, w_std=0.05)
    m[-1] = 1
    x[-1] = V - 1
    lp, ent = O.token_logprobs(O.widen_bf16(h), O.widen_bf16(W), x, m)
    a, e = getattr(molt, call)(bf(h), bf(W), t(x), t(m))
    torch.cuda.synchronize()
    assert molt.device_status() == 0
    # products of bf16 are exact in fp32, sums of H of them and of V exponentials
    # are off by at most a few times (H + V / 256) 2^-24 of terms of order 10
    bound = min(LOGP_ATOL, 40 * (H + V / 256 + 64) * 2.0 ** -24)
    assert np.abs(np_(a) - lp).max() <= bound
    assert np.abs(np_(e) - ent).max() <= bound
    assert (np_(a)[m == 0] == 0).all() and (np_(e)[m == 0] == 0).all()


# a NaN in one column reaches every row, one in a hidden row that row alone, whichever
# half of a tile and whichever of the vocab splits (T = 20: one for each tile) holds it
@pytest.mark.parametrize("T,col", [(20, 3), (20, 2000), (300, 130), (300, 4100)])
@pytest.mark.parametrize("call", ["token_logprobs", "token_logprobs_noalloc", "vp"])
def test_nan_reaches_the_row(T, col, call):
    H, V, bad = 256, 4300, T // 2
    rng = np.random.default_rng(T + col)
    h, W, x, _ = random_problem(rng, T, H, V, w_std=0.05)
    x[x == col] = col - 1
    h, W, x = bf(h), bf(W), t(x)

    def run(h, W):
        if call != "vp":
            return getattr(molt, call)(h, W, x)
        cut = 2048
        parts = torch.stack([molt.vp_partials(h, W[:cut].contiguous(), x, 0),
                             molt.vp_partials(h, W[cut:].contiguous(), x, cut)])
        z = torch.zeros(T, device="cuda")
        out = molt.vp_loss(parts, z, z)
        return out["logp"], out["entropy"]

    h2, W2 = h.clone(), W.clone()
    h2[bad, 7] = float("nan")
    W2[col, 9] = float("nan")
    lp0, e0 = run(h, W)
    lp1, e1 = run(h, W2)
    assert torch.isnan(lp1).all() and torch.isnan(e1).all()
    lp2, e2 = run(h2, W)
    torch.cuda.synchronize()
    # the shard merge reports a NaN target logit as a target in no shard instead
    assert torch.isnan(e2[bad])
    assert molt.device_status() != 0 if call == "vp" else torch.isnan(lp2[bad])
    keep = torch.arange(T, device="cuda") != bad
    assert torch.equal(lp2[keep], lp0[keep]) and torch.equal(e2[keep], e0[keep])
