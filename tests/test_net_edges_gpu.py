"""The network's elementwise kernels at the shapes where their splits can go
wrong: output layers of 1 to 16 channels (one kernel each) and channel counts
that do and do not let a warp fold its bias sums by shuffles (48 and 80 are 6
and 10 groups of 8).

Gradients: both sides take the same BF16 activations (the network oracle with
BF16 storage); what differs is the order of FP32 sums, 2^-24 sqrt(K) of the
summed magnitudes, and sparse one-unit flips of stored BF16 values: 4 units
of 2^-8 of each layer's largest value."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import unet
from paper_2011_00814_gb300 import build, gpe2p

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,channels,out_ch", [(1, [16], 1), (2, [48, 80], 2), (1, [32], 3), (2, [16, 64], 5),
                                                    (1, [48], 7), (2, [80, 96], 8), (1, [64], 11), (2, [32, 48], 16)])
def test_head_and_bias_gradients_match_oracle(levels, channels, out_ch):
    import torch
    build.build()
    rng = np.random.default_rng(5 + out_ch)
    b, h, w = 3, 22, 18
    x = rng.normal(size=(b, h, w, 4)).astype(np.float32)
    t = (0.5 * rng.normal(size=(b, h, w, out_ch))).astype(np.float32)
    convs, (hc, ho) = unet.layer_shapes(levels, channels, 4, out_ch)
    with gpe2p.Net(levels, channels, 4, out_ch, h, w, b, seed=11) as net:
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
    parts += [("head", slice(o, o + ho * hc)), ("head bias", slice(o + ho * hc, o + ho * hc + ho))]
    lref, gref = unet.loss_and_gradient(pref, x.astype(np.float64), t.astype(np.float64), levels, channels, 4, out_ch,
                                        bf16=True)
    assert abs(loss - lref) <= 1e-3 * lref
    for name, s in parts:
        assert np.max(np.abs(g[s] - gref[s])) <= 4.0 * 2.0 ** -8 * np.max(np.abs(gref[s])), name
