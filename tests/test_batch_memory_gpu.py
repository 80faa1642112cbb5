"""An instance of a batch holds 17 fields of its padded grid, in FP64 too, where the
flow stages keep their frozen terms in fields that are free at that time."""
from __future__ import annotations

import pytest
import torch

from paper_2011_00814_gb300 import build, gpe2p, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [32, 64])
def test_device_memory_of_a_batch(precision):
    build.build()
    nx = ny = 1024                                    # rows of 1024 values need no padding
    prms = []
    for k in range(4):
        prm = inputs.base_params(2, nx, ny, dx=0.5, dt=0.02, cs=1.2, rhoL=1.0, rhoG=0.2, etaL=0.05, etaG=0.01,
                                 rho_ref=0.6, sigma=0.03, M=0.02, W=2.0, g=(0.0, -0.02, 0.0),
                                 bc=("periodic", "noslip", "periodic"), ch_advection=k % 2)
        prm["precision"] = precision
        prms.append(prm)
    with gpe2p.Batch(prms[:1]):
        pass                                          # the context and the modules are loaded
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    with gpe2p.Batch(prms):
        used = free0 - torch.cuda.mem_get_info()[0]
    field = nx * ny * precision // 8
    # besides the fields: the FP64 staging of one instance, the work tables, the
    # scratch of the diagnostics and the graphs: below 16 MiB and a field's size
    assert used <= 4 * 17 * field + nx * ny * 8 + (16 << 20), used / (4 * field)
