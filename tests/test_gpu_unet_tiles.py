"""The U-Net convolution and weight-gradient kernels at the edges of their
tiles (16 x 8/16/32 and 8 x 16 pixels with a halo), channel chunks, output
channel blocks and pixel splits, against the FP64 oracle on the same
BF16-rounded inputs.

Convolution: FP32 accumulation of K = 9 cin products, then one BF16 rounding.
Against the oracle's unrounded value that is half a BF16 step (at most 2^-8 of
the value) plus the accumulation error, K 2^-24 times the sum of the products'
magnitudes, twice that for the bias and the value's own error in the first term.  Weight gradient: FP32 sums of P = B H W products,
so P 2^-24 times the sum of the magnitudes, per entry.
"""
import numpy as np
import pytest
import torch

from oracle import unet as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def un():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14189_gb300 import unet
    return unet


def bf(x):
    return torch.tensor(np.asarray(x, dtype=np.float32)).to(torch.bfloat16).cuda()


def host(t):
    return t.float().cpu().numpy().astype(np.float64)


CASES = [  # B, H, W, cin, cout
    (1, 8, 16, 32, 32),      # one tile, half of it off the image
    (3, 24, 16, 96, 160),    # 32-channel chunks; rows not a multiple of the tile's
    (1, 9, 256, 32, 64),     # odd rows
    (1, 8, 16, 192, 192),    # several input blocks, the last one short
    (2, 12, 32, 224, 224),   # seven 32-channel chunks
    (1, 6, 64, 64, 96),
    (1, 8, 16, 544, 224),    # input tile staged again for every tap
    (1, 16, 128, 512, 256),
]


@pytest.mark.parametrize("op", [0, 1, 2])
@pytest.mark.parametrize("case", CASES)
def test_convolution(un, case, op):
    B, H, W, ci, co = case
    rng = np.random.default_rng(sum(case) + op)
    x = U.bf16(rng.standard_normal((B, H, W, ci)))
    w = U.bf16(rng.standard_normal((co, 3, 3, ci)) * np.sqrt(2.0 / (9 * ci)))
    b = U.fp32(rng.standard_normal(co) * 0.1) if op == un.OP_RELU else np.zeros(co)
    m = U.bf16(rng.standard_normal((B, H, W, co)))
    out = un.conv3x3(bf(x), bf(w.reshape(co, 9, ci)),
                     torch.tensor(b, dtype=torch.float32).cuda() if op == un.OP_RELU else None,
                     op=op, mask=bf(m) if op == un.OP_MASK else None)
    ref, mag = U.conv3x3(x, w, b), U.conv3x3(np.abs(x), np.abs(w), np.abs(b))
    if op == un.OP_RELU:
        ref = np.maximum(ref, 0.0)
    if op == un.OP_MASK:
        ref = np.where(m > 0, ref, 0.0)
    err = np.abs(host(out) - ref)
    assert (err <= 2.0 ** -8 * np.abs(ref) + 9 * ci * 2.0 ** -24 * mag * 2).all()


@pytest.mark.parametrize("case", CASES)
def test_weight_gradient(un, case):
    B, H, W, ci, co = case
    rng = np.random.default_rng(sum(case))
    x = U.bf16(rng.standard_normal((B, H, W, ci)))
    dy = U.bf16(rng.standard_normal((B, H, W, co)))
    got = un.conv3x3_wgrad(bf(x), bf(dy)).cpu().numpy().astype(np.float64)
    xp = np.pad(x, ((0, 0), (1, 1), (1, 1), (0, 0)))
    d = dy.reshape(-1, co)
    for tap in range(9):
        xs = xp[:, tap // 3:tap // 3 + H, tap % 3:tap % 3 + W].reshape(-1, ci)
        err = np.abs(got[:, tap] - d.T @ xs)
        assert (err <= B * H * W * 2.0 ** -24 * (np.abs(d).T @ np.abs(xs))).all(), tap
