"""The 3D kernels at the sizes where their tiles can go wrong: the flow tile is
30 cells wide and overlaps its neighbour by a lane, so 29, 30, 31 and 61 wide; one
cell or one plane; a last row or plane alone in its tile; walls beside periodic
sides, whose ghosts come from shared memory; conservative advection, both time
schemes and each stencil.

Reference: the FP64 oracle.  Three stages of sums of up to forty terms round to
eps x 40 x 3 of the largest term per step; the largest term of the pressure
rate, rho c_s^2 div u dt, is below 10 times the pressure compared.  Three steps:
FP64 4e-13 x 10, held to 1e-11 as in 2D; FP32 (eps = 2^-24) 2.2e-5 x 10 = 2.2e-4 of
each field's largest value."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2011_00814_gb300 import build, gpe2p, inputs

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (1, 7, 5), (29, 9, 3), (30, 8, 1), (31, 17, 6), (61, 5, 33), (64, 33, 18)]
BC = [("periodic", "periodic", "periodic"), ("noslip", "freeslip", "periodic"), ("periodic", "noslip", "freeslip"),
      ("freeslip", "periodic", "noslip")]
FORMS = {"rk2": dict(), "rk4": dict(ch_scheme=4), "conservative": dict(ch_advection=1),
         "q15-bare": dict(iso=15, bulk_visc=0, p_average=0), "q27": dict(iso=27, ch_scheme=4)}


@pytest.mark.parametrize("precision,tol", [(64, 1e-11), (32, 2.2e-4)])
@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("size,bc", [(s, BC[(i + j) % 4]) for i, s in enumerate(SIZES) for j in (0, 1)])
def test_steps_match_oracle(size, bc, form, precision, tol):
    build.build()
    prm = inputs.base_params(3, *size, dx=0.5, dt=0.02, cs=1.2, rhoL=1.0, rhoG=0.3, etaL=0.05, etaG=0.01,
                             rho_ref=0.6, sigma=0.03, M=0.02, W=2.0, g=(0.01, -0.02, 0.005), bc=bc)
    prm.update(precision=precision, **FORMS[form])
    f = inputs.random_fields(prm, seed=8)
    n = 3
    with gpe2p.Solver(prm) as s:
        s.init_fields(f)
        s.advance(n)
        got = s.read_fields()
    st = oracle.init_state(prm, f["phi"], f["p"], f["u"], f["v"], f["w"])
    ref = oracle.step(prm, st, n)
    for k in ("phi", "u", "v", "w", "p"):
        assert np.max(np.abs(got[k] - ref[k])) <= tol * max(np.max(np.abs(ref[k])), 1e-2), k
