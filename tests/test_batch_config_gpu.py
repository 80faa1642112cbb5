"""The tile that a batch reports is the tile that runs."""
from __future__ import annotations

import pytest

from paper_2011_00814_gb300 import build, gpe2p, inputs

pytestmark = pytest.mark.gpu

SWEEPS = ((32, 8), (64, 4), (16, 16))
SHORT, TALL = (26, 12), (26, 28)                          # tiles of the fused flow pass


@pytest.mark.parametrize("precision,conservative,n,persistent,tiles", [
    (32, 0, 2, 0, (SHORT,)), (32, 0, 2, 1, (SHORT,)),
    (32, 0, 20, 0, (TALL,)), (32, 0, 20, 1, (SHORT,)),    # 20 x 50 tall tiles of 256 x 128
    (32, 1, 2, 0, SWEEPS), (64, 0, 2, 0, SWEEPS), (64, 1, 2, 1, SWEEPS)])
def test_reported_tile(precision, conservative, n, persistent, tiles):
    build.build()
    prm = inputs.base_params(2, 256, 128, dx=0.5, dt=0.02, cs=1.2, rhoL=1.0, rhoG=0.25, etaL=0.05, etaG=0.01,
                             rho_ref=0.6, sigma=0.03, M=0.02, W=2.0, g=(0.0, 0.0, 0.0),
                             bc=("periodic", "periodic", "periodic"))
    prm["precision"] = precision
    with gpe2p.Batch([prm] * (n - 1) + [dict(prm, ch_advection=conservative)]) as b:
        b.fault(gpe2p.FAULT_FORCE_PERSISTENT, persistent)
        c = b.config()
    assert c["tile"] in tiles and c["persistent"] == bool(persistent)
