"""The cluster backward (csrc/lmhead_bwd4.cu) at sizes that select it: H = 128, H = 384
below 512 rows, whose last job is 128 columns wide, and reproducible calls of many
columns.  Raster and reproducible schedule, the latter over several groups of four token
quads and more vocab blocks than clusters, and the vocabulary split with the single-CTA
kernel."""
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


def _problem(T, H, V, deterministic):
    assert molt.backward_plan(T, H, V, deterministic)["kernel"] == "lmhead_bwd_quad_kernel"
    rng = np.random.default_rng(T + H + V)
    h, W, x, m = random_problem(rng, T, H, V, mask_frac=0.1, w_std=0.05)
    m[0] = 1
    x[:32] = rng.integers(max(0, V - 500), V, min(T, 32))   # in the last block
    adv = rng.standard_normal(T).astype(np.float32)
    h64, W64 = O.widen_bf16(h), O.widen_bf16(W)
    b = behavior_from_oracle(h64, W64, x, 0.3, 0.2, 0.28, T)
    ref = O.policy_loss(h64, W64, x, b.astype(np.float64), adv.astype(np.float64), m, 0.2, 0.28)
    ref["_adv"] = adv.astype(np.float64)
    return (bf(h), bf(W), t(x), t(b), t(adv), t(m), 0.2, 0.28), ref


def _check(out, ref):
    torch.cuda.synchronize()
    assert molt.device_status() == 0
    assert_loss_close(float(out["loss"].item()), ref)
    assert_grad_close(np_(out["dhidden"]), ref["dH"], "dhidden")
    assert_grad_close(np_(out["dW"]), ref["dW"], "dW")


@pytest.mark.parametrize("T,H,V", [(1, 128, 7), (513, 128, 1025), (5000, 128, 9000), (400, 384, 3000), (511, 384, 19000)])
def test_raster(T, H, V):
    args, ref = _problem(T, H, V, False)
    _check(molt.policy_loss_fwd_bwd(*args), ref)


# (5000, 128, 9000): three groups of four token quads; 18, 38 and 51 vocab blocks for nine
# clusters a token quad; (700, 384, 26000): the same with a 128-column last job; (600, 512, 25600): the
# least V of the rule
@pytest.mark.parametrize("T,H,V", [(513, 128, 1025), (5000, 128, 9000), (511, 384, 19000), (700, 384, 26000),
                                   (600, 512, 25600)])
def test_reproducible_whatever_the_cluster_count(T, H, V):
    args, ref = _problem(T, H, V, True)
    outs = [molt.policy_loss_fwd_bwd_ex(*args, deterministic=True, det_clusters=n) for n in (0, 0, 16, 8, 4)]
    _check(outs[0], ref)
    for o in outs[1:]:
        for k in ("dW", "dhidden"):
            assert torch.equal(o[k].view(torch.uint8), outs[0][k].view(torch.uint8)), k


@pytest.mark.parametrize("V", [18986, 19243])
def test_vocabulary_split(V):
    """36 whole blocks go to the 36 clusters of a GB300 and the last 554 or 811 columns to
    the single-CTA kernel on the SMs that no cluster can use; without them the call has
    one launch fewer."""
    T, H = 700, 128
    args, ref = _problem(T, H, V, False)
    n0 = molt.kernel_launches()
    out = molt.policy_loss_fwd_bwd(*args)
    n_split = molt.kernel_launches() - n0
    _check(out, ref)
    assert_grad_close(np_(out["dW"])[V - 1024:], ref["dW"][V - 1024:], "dW last columns")
    x = torch.clamp(args[2], max=18431)
    n0 = molt.kernel_launches()
    molt.policy_loss_fwd_bwd(args[0], args[1][:18432], x, *args[3:])
    n_plain = molt.kernel_launches() - n0
    torch.cuda.synchronize()
    assert molt.device_status() == 0
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert n_split == n_plain + 1
