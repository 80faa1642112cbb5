"""The 2D FP64 flow stage at the sizes where its tiles can go wrong (one cell,
one row, a cell past a tile edge, each of its three tile shapes), with every mix of
walls, without averaging or bulk viscosity and in the axisymmetric form: the
terms frozen over the stages are written by one stage and read by the next, past the
domain's high end from the wrapped or mirrored cells.

Reference: the FP64 oracle.  Three stages of sums of up to forty terms round to
about 2^-53 x 40 x 3 = 1.3e-14 of the largest term per step; the largest term of
the pressure rate, rho c_s^2 div u dt, is below 10 times the pressure compared,
so five steps stay below 1e-12 x 10 of each field's largest value."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2011_00814_gb300 import build, gpe2p, inputs

pytestmark = pytest.mark.gpu

BC = [("periodic", "periodic"), ("noslip", "freeslip"), ("periodic", "noslip"), ("freeslip", "periodic")]
SIZES = [(1, 1), (1, 9), (8, 4), (9, 5), (17, 31), (64, 64), (161, 129), (400, 300)]


@pytest.mark.parametrize("bc", BC)
@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("form", ["plain", "bare", "axisym"])
def test_fp64_steps_match_oracle(size, bc, form):
    if form == "axisym" and bc[0] == "periodic":
        pytest.skip("the axisymmetric form has an outer wall")
    build.build()
    prm = inputs.base_params(2, *size, dx=0.5, dt=0.02, cs=1.2, rhoL=1.0, rhoG=0.3, etaL=0.05, etaG=0.01,
                             rho_ref=0.6, sigma=0.03, M=0.02, W=2.0,
                             g=(0.0 if form == "axisym" else 0.01, -0.02, 0.0), bc=bc + ("periodic",))
    prm.update(precision=64)
    if form == "bare":
        prm.update(bulk_visc=0, p_average=0)
    if form == "axisym":
        prm.update(axisym=1)
    f = inputs.random_fields(prm, seed=8)
    n = 5
    with gpe2p.Solver(prm) as s:
        s.init_fields(f)
        s.advance(n)
        got = s.read_fields()
    st = oracle.init_state(prm, f["phi"], f["p"], f["u"], f["v"])
    ref = oracle.step(prm, st, n)
    for k in ("phi", "u", "v", "p"):
        assert np.max(np.abs(got[k] - ref[k])) <= 1e-11 * max(np.max(np.abs(ref[k])), 1e-2), k
