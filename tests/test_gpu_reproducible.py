"""The reproducible loss call gives the bits that are on record
(tests/golden/reproducible.txt): a run that is resumed with another version of the
library goes on as if nothing had changed.  The records were taken on a GB300 from
the library as it was when one thread folded a row's 256-column tiles one after the
other and the cluster kernel alone did the backward, 512 tokens and columns at a time.

Inputs are made of integer arithmetic and exact conversions, the same on every
machine and with every numpy.
"""
import hashlib
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2607_21653_gb300 as molt  # noqa: E402

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "reproducible.txt")

# the cluster kernel (H = 128; H = 384 below 512 rows and at 30000 columns, whose last
# job is 128 columns)
# and the one over chunks: one row, a remainder of one row in the second term, several
# terms and chunks in both directions, chunks of 16 x 16 tiles
SHAPES = [(700, 128, 5000), (400, 384, 3000), (1, 256, 7), (513, 512, 4133), (900, 384, 3000), (2100, 640, 20000),
          (5000, 256, 9000), (769, 256, 8200), (700, 384, 30000), (4700, 1536, 40000), (4300, 2176, 8300)]
# the surrogate alone; with KL, entropy bonus and sequence gate, added to a dW;
# gradients so small that most of them are subnormal
VARIANTS = ("plain", "extended", "subnormal")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    molt.build()
    molt.load()


def _uniform(n, seed):
    """n values in [0, 1), multiples of 2^-24: the splitmix64 sequence."""
    with np.errstate(over="ignore"):
        z = (np.arange(1, n + 1, dtype=np.uint64) + np.uint64(seed << 40)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z ^= z >> np.uint64(31)
    return (z >> np.uint64(40)).astype(np.float32) * np.float32(2.0 ** -24)


def _bell(n, seed, scale):
    """Mean 0, standard deviation `scale` (a power of two): the sum of three uniforms, doubled."""
    u = sum(_uniform(n, 4 * seed + i) for i in range(3)) - np.float32(1.5)
    return u * np.float32(2 * scale)


def _call(T, H, V, variant):
    dev = "cuda"
    bf = lambda a, *shape: torch.from_numpy(a).to(dev).view(*shape).to(torch.bfloat16)
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    h, W = bf(_bell(T * H, 1, 1.0), T, H), bf(_bell(V * H, 2, 2.0 ** -5), V, H)
    x = up((_uniform(T, 20) * V).astype(np.int32))
    m = up((np.arange(T) % 7 != 3).astype(np.uint8))
    b = up(np.float32(-np.floor(np.log(V) * 64) / 64) + _bell(T, 6, 0.125))
    adv = _bell(T, 7, 1.0)
    kw = {}
    if variant == "extended":
        kw = dict(kl_coef=0.0625, ref_logp=b + 0.125, entropy_coef=0.015625, gate_lo=0.5, gate_hi=2.0,
                  seq_of_token=up((np.arange(T) // 96).astype(np.int32)), accumulate_dW=True,
                  dW=up(_bell(V * H, 8, 2.0 ** -10).reshape(V, H)))
    if variant == "subnormal":
        adv *= np.float32(2.0 ** -110)
    return molt.policy_loss_fwd_bwd_ex(h, W, x, b, up(adv), m, 0.25, 0.25, deterministic=True, **kw)


def digests(T, H, V, variant):
    out = _call(T, H, V, variant)
    torch.cuda.synchronize()
    assert molt.device_status() == 0
    return " ".join(k + "=" + hashlib.sha256(out[k].contiguous().view(torch.uint8).cpu().numpy().tobytes()).hexdigest()[:12]
                    for k in ("loss", "dhidden", "dW", "logp", "entropy", "token_loss", "stats"))


@pytest.mark.parametrize("variant", VARIANTS)
@pytest.mark.parametrize("T,H,V", SHAPES)
def test_the_bits_on_record(T, H, V, variant):
    with open(GOLDEN) as f:
        lines = dict(line.strip().split(": ", 1) for line in f if ": " in line and not line.startswith("#"))
    assert digests(T, H, V, variant) == lines[f"{T} {H} {V} {variant}"]
