"""2D problems with the RK4 Cahn-Hilliard scheme: in FP32 the fused flow pass is
followed by the stages one by one, in FP64 the RK4 accumulator and a stage buffer hold
the flow step's frozen terms until the stages begin.  Grids of every FP64 tile and
both FP32 tile heights, advective and conservative form, compensated phi.

Reference: the FP64 oracle.  FP64: sums of up to forty terms, (3 + 4) stages a step,
2^-53 x 40 x 7 = 3e-14 of the largest term, at most 10 times the field: 1e-11 for four
steps leaves a factor of ten.  FP32: 2^-24 x (3 + 4) stages x 4 steps x 8 (sums of up
to a dozen terms) = 1.4e-5."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2011_00814_gb300 import build, gpe2p, inputs

pytestmark = pytest.mark.gpu

BC = [("periodic", "periodic"), ("noslip", "freeslip"), ("periodic", "noslip")]


@pytest.mark.parametrize("precision,tol", [(64, 1e-11), (32, 1.4e-5)])
@pytest.mark.parametrize("form", ["advective", "conservative", "compensated"])
@pytest.mark.parametrize("bc", BC)
@pytest.mark.parametrize("size", [(1, 9), (27, 13), (161, 129), (420, 1000)])
def test_rk4_steps_match_oracle(size, bc, form, precision, tol):
    if form == "compensated" and precision == 64:
        pytest.skip("FP64 keeps phi in one word")
    build.build()
    prm = inputs.base_params(2, *size, dx=0.5, dt=0.02, cs=1.2, rhoL=1.0, rhoG=0.3, etaL=0.05, etaG=0.01,
                             rho_ref=0.6, sigma=0.03, M=0.02, W=2.0, g=(0.01, -0.02, 0.0), bc=bc + ("periodic",))
    prm.update(precision=precision, ch_scheme=4, ch_advection=int(form == "conservative"))
    f = {k: v.astype(np.float32).astype(np.float64) for k, v in inputs.random_fields(prm, seed=6).items()}
    n = 4
    with gpe2p.Solver(prm) as s:
        s.set_phi_accumulation(gpe2p.PHI_ACC_COMPENSATED if form == "compensated" else gpe2p.PHI_ACC_FP32)
        s.init_fields(f)
        s.advance(n)
        got = s.read_fields()
    ref = oracle.step(prm, oracle.init_state(prm, f["phi"], f["p"], f["u"], f["v"]), n)
    for k in ("phi", "u", "v", "p"):
        assert np.max(np.abs(got[k] - ref[k])) <= tol * max(np.max(np.abs(ref[k])), 1e-2), k
