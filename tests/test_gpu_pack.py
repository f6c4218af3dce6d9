"""The row packing on both sides of the forward (csrc/rows.cu: pack_kernel,
finish_kernel) where it can go wrong: fewer rows than blocks, one more or less than
8 blocks on each of 152 SMs, more than 256 rows a block, a mask that starts at any
byte and holds any nonzero value, no active row, only the last one, no mask."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2607_21653_gb300 as molt  # noqa: E402
from oracle import molt_oracle as O  # noqa: E402
from workloads import random_problem  # noqa: E402

from parity import LOGP_ATOL, assert_grad_close, assert_loss_close, behavior_from_oracle, bf, np_, t  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    molt.build()
    molt.load()


@pytest.mark.parametrize("T,H,mask", [
    (1, 256, "none"), (1215, 256, "random"), (1216, 64, "all"), (1217, 256, "random"), (2433, 256, "last"),
    (5000, 256, "zero"), (5000, 128, "zero"), (39000, 256, "random"), (311297, 64, "all"), (330000, 64, "random"),
    (311400, 64, "none")])
def test_rows_are_packed_in_order(T, H, mask):
    V, rng = 9, np.random.default_rng(T + H)
    h, W, x, _ = random_problem(rng, T, H, V, w_std=0.05)
    # every nonzero byte is an active row
    m = rng.integers(1, 256, size=T).astype(np.uint8)
    if mask == "random":
        m[rng.random(T) < 0.4] = 0
    elif mask == "last":
        m[:-1] = 0
    elif mask == "zero":
        m[:] = 0
    on = (m != 0).astype(np.uint8)
    adv = rng.standard_normal(T).astype(np.float32)
    adv[rng.random(T) < 0.3] = 0
    adv[-1] = 1.5
    h64, W64 = O.widen_bf16(h), O.widen_bf16(W)
    b = behavior_from_oracle(h64, W64, x, 0.3, 0.2, 0.28, T)
    ref = O.policy_loss(h64, W64, x, b.astype(np.float64), adv.astype(np.float64), on, 0.2, 0.28, denom=float(T),
                        block=4096)
    ref["_adv"] = adv.astype(np.float64)
    fixed = (bf(h), bf(W), t(x), t(b), t(adv))
    buf = torch.empty(T + 16, dtype=torch.uint8, device="cuda")
    for shift in (0, 1, 15):
        if mask == "none":
            dm = None
        else:
            dm = buf[shift:shift + T]
            dm.copy_(t(m))
        dW = torch.full((V, H), float("nan"), device="cuda")
        out = molt.policy_loss_fwd_bwd(*fixed, dm, 0.2, 0.28, denom=float(T), dW=dW)
        torch.cuda.synchronize()
        assert molt.device_status() == 0
        st = molt.stats_dict(out["stats"])
        assert st["n_active"] == int(on.sum())
        assert st["n_grad_rows"] == int(np.count_nonzero(ref["coef"]))
        assert_loss_close(float(out["loss"].item()), ref)
        assert_grad_close(np_(out["dhidden"]), ref["dH"], "dhidden")
        assert_grad_close(np_(out["dW"]), ref["dW"], "dW")
        off = on == 0
        assert np.abs(np_(out["logp"]) - ref["logp"]).max() <= LOGP_ATOL
        for k in ("logp", "entropy", "token_loss"):
            assert (np_(out[k])[off] == 0).all()
        assert (np_(out["dhidden"])[ref["coef"] == 0] == 0).all()
        if mask == "none":
            break
