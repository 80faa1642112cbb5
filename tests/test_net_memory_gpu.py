"""A network holds the tensors that its passes use and no others: the output of an
encoder level and its gradient lie in the decoder's concatenated tensor."""
from __future__ import annotations

import pytest
import torch

from paper_2011_00814_gb300 import build, gpe2p

pytestmark = pytest.mark.gpu


def test_device_memory_of_a_network():
    build.build()
    ch, n, batch = [64, 128, 256], 512, 4
    with gpe2p.Net(1, [16], 5, 5, 32, 32, 1):
        pass                                              # the context and the modules are loaded
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    with gpe2p.Net(3, ch, 5, 5, n, n, batch):
        used = free0 - torch.cuda.mem_get_info()[0]
    px = [batch * (n >> l) ** 2 for l in range(3)]
    # BF16 tensors, value and gradient: the padded input; each level's first output; the
    # last level's second; pooled, upsampled, concatenated and the decoder's two outputs
    act = 16 * px[0] + sum(c * p for c, p in zip(ch, px)) + ch[2] * px[2]
    for l in range(2):
        act += ch[l] * px[l + 1] + ch[l + 1] * px[l] + 4 * ch[l] * px[l]
    # pre-activations of the convolutions, and the largest as scratch
    pre = sum(2 * c * p for c, p in zip(ch, px)) + sum(3 * ch[l] * px[l] for l in range(2)) + ch[0] * px[0]
    weights = 32 << 20                                    # 1.9 M weights in FP32 (4) and BF16 (4)
    pages = 64 * (2 << 20)                                # an allocation's last 2 MiB page
    assert used <= 4 * act + 2 * pre + 40 * px[0] + weights + pages, (used, 4 * act + 2 * pre)
