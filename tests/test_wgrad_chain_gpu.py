"""The length of the weight gradient's FP32 sums, through a network whose
products are known exactly.  The first convolution copies its input (a centre tap
of 1, activations where SiLU is the identity or zero in BF16), the second has zero
weights and the head weight 1, so that dZ of the second is the target over the number
of outputs in BF16 and its weight gradient is the sum over pixels of X(p + tap) dZ(p),
all terms positive, factors of 8 significant bits.

Bound: the tensor cores' FP32 accumulation may truncate, 2^-23 of the partial sum for
each of the K steps of 16 pixels.  Sums of at most 2048 pixels are 128 steps, whose
partial sums grow evenly: 64.5 x 2^-23 of the sum; the parts are added by FP32
atomics, 2^-24 of the partial sum each: (m + 1) / 2 x 2^-24 for m of them, where
a part may be as short as half of the longest."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2011_00814_gb300 import build, gpe2p

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c,h,w,b", [(32, 256, 256, 8), (256, 128, 128, 8), (1024, 64, 64, 4), (48, 72, 200, 8)])
def test_long_sums_are_cut(c, h, w, b):
    import torch
    build.build()
    rng = np.random.default_rng(c)
    bf16 = lambda a: torch.from_numpy(a.astype(np.float32)).bfloat16().float().numpy()
    x = np.where(rng.random((b, h, w, 4)) < 0.3, np.float32(-100), bf16(32 * 2 ** rng.uniform(0, 3, (b, h, w, 4))))
    k = bf16(2 ** rng.uniform(-3, 3, (b, h, w, 1)))
    n = b * h * w
    with gpe2p.Net(1, [c], 4, 1, h, w, b, seed=1) as net:
        p = np.zeros(net.nparam, np.float32)
        p[:c * 9 * 16].reshape(c, 9, 16)[np.arange(c), 4, np.arange(c) % 4] = 1.0
        p[-(c + 1):-1] = 1.0
        net.set_params(p)
        _, g = net.gradients(torch.from_numpy(x).cuda(), torch.from_numpy(-k).cuda(), b)
    o = c * 9 * 16 + c
    got = g[o:o + c * 9 * c].reshape(c, 9, c).astype(np.float64)
    X = torch.from_numpy(np.maximum(x, 0)).double().cuda().permute(0, 3, 1, 2)
    inv = float(np.float32(1.0) / np.float32(n))
    dy = (torch.from_numpy(2 * k).cuda() * np.float32(inv)).bfloat16()     # 2 d / n, stored in BF16
    dz = (dy.float() * 0.5).bfloat16().double().permute(0, 3, 1, 2)        # SiLU'(0) = 1/2
    ref = np.stack([(torch.roll(X, (-i, -j), (2, 3)) * dz).sum((0, 2, 3)).cpu().numpy()
                    for i in (-1, 0, 1) for j in (-1, 0, 1)])
    ref = ref[:, np.arange(c) % 4]
    parts = 2 * -(-n // 2048)
    bound = 64.5 * 2.0 ** -23 + (parts + 1) / 2 * 2.0 ** -24
    assert np.max(np.abs(got - ref[None]) / ref[None]) <= bound
