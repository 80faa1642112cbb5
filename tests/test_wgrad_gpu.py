"""The tcgen05 weight gradient at the shapes where its tiling can go wrong:
images smaller than its 16 x 8 pixel tile, images the tiles overhang, channel
counts that take each of its block sizes (16, 32, 64, 128, and 48 = 3 x 16), the
upsampled input of the decoder, and more tiles than CTAs.

Both sides take the same BF16 activations and dZ (the network oracle with
BF16 storage, see test_net_gpu): what differs is the FP32 against FP64 sum of
the products, about 2^-24 sqrt(K) of the summed magnitudes, and sparse
one-unit BF16 flips of stored values; the bound on every layer's weight and
bias gradient is the one derived there, 4 units of 2^-8 of the layer's largest."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import unet
from paper_2011_00814_gb300 import build, gpe2p

pytestmark = pytest.mark.gpu

SHAPES = [(1, [16], 1, 1, 1), (1, [64], 17, 9, 2), (2, [16, 32], 6, 10, 3), (2, [32, 64], 34, 14, 1),
          (2, [48, 96], 18, 26, 2), (2, [64, 128], 32, 8, 2), (3, [32, 16, 64], 36, 20, 1), (1, [32], 200, 136, 3),
          (2, [32, 128], 20, 12, 2), (2, [128, 256], 18, 14, 1)]


@pytest.mark.parametrize("levels,channels,h,w,b", SHAPES)
def test_weight_gradients_match_oracle(levels, channels, h, w, b):
    import torch
    build.build()
    rng = np.random.default_rng(21)
    x = rng.normal(size=(b, h, w, 4)).astype(np.float32)
    t = (0.5 * rng.normal(size=(b, h, w, 4))).astype(np.float32)
    convs, (hc, ho) = unet.layer_shapes(levels, channels, 4, 4)
    with gpe2p.Net(levels, channels, 4, 4, h, w, b, seed=11) as net:
        p = net.get_params()
        p[-(ho * hc + ho):] = 0.3 * rng.normal(size=ho * hc + ho)
        net.set_params(p)
        loss, g = net.gradients(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), b)
    pref, o, parts = p.astype(np.float64), 0, []
    for name, cin, cout, taps in convs:
        n = cout * taps * cin
        pref[o:o + n] = unet.round_bf16(p[o:o + n])
        parts += [(name, slice(o, o + n)), (name + " bias", slice(o + n, o + n + cout))]
        o += n + cout
    lref, gref = unet.loss_and_gradient(pref, x.astype(np.float64), t.astype(np.float64), levels, channels, 4, 4,
                                        bf16=True)
    assert abs(loss - lref) <= 1e-3 * lref
    for name, s in parts:
        assert np.max(np.abs(g[s] - gref[s])) <= 4.0 * 2.0 ** -8 * np.max(np.abs(gref[s])), name
