"""The tall tiles of the fused 2D FP32 passes (grids and batches with two or more for
every SM): every mix of walls, the axisymmetric form and the compensated phi
accumulation of a single problem against the FP64 oracle, and a batch of planar,
axisymmetric and conservative instances, one launch per pass, against single
problems with the short tiles, bit for bit.

Bound against the oracle: FP32 rounding of q + dt L is 2^-24 of the field per stage,
times (3 + 2) stages a step and eight (sums of up to a dozen terms): for two
steps 5e-6, held to 1e-5; phi's rounding enters mu through kappa lap ~ 16 kappa /
dx^2, which scales its bound."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2011_00814_gb300 import build, gpe2p, inputs

pytestmark = pytest.mark.gpu

BC = [("periodic", "periodic"), ("noslip", "freeslip"), ("freeslip", "noslip"), ("periodic", "noslip")]


def problem(nx, ny, bc, axisym=0, seed=3, **kw):
    prm = inputs.base_params(2, nx, ny, dx=0.5, dt=0.02, cs=1.2, rhoL=1.0, rhoG=0.3, etaL=0.05, etaG=0.01,
                             rho_ref=0.6, sigma=0.03, M=0.02, W=2.0, g=(0.0 if axisym else 0.01, -0.02, 0.0),
                             bc=bc + ("periodic",))
    prm.update(precision=32, axisym=axisym, **kw)
    f = inputs.random_fields(prm, seed=seed)
    return prm, {k: v.astype(np.float32).astype(np.float64) for k, v in f.items()}


@pytest.mark.parametrize("mode", [gpe2p.PHI_ACC_FP32, gpe2p.PHI_ACC_COMPENSATED])
@pytest.mark.parametrize("bc", BC)
@pytest.mark.parametrize("size", [(1200, 300), (417, 1001)])
def test_tall_single_problem_matches_oracle(size, bc, mode):
    build.build()
    for axisym in (0, 1):
        if axisym and bc[0] == "periodic":
            continue
        prm, f = problem(*size, bc, axisym)
        with gpe2p.Solver(prm) as s:
            s.set_phi_accumulation(mode)
            s.init_fields(f)
            s.advance(2)
            got = s.read_fields()
        ref = oracle.step(prm, oracle.init_state(prm, f["phi"], f["p"], f["u"], f["v"]), 2)
        for k in ("phi", "u", "v", "p"):
            scale = max(np.max(np.abs(ref[k])), 1e-2)
            assert np.max(np.abs(got[k] - ref[k])) <= 1e-5 * scale, (axisym, k)
        assert np.max(np.abs(got["mu"] - ref["mu"])) <= 1e-5 * 16.0 * 0.75 / 0.25, (axisym, "mu")


def test_tall_batch_matches_single_problems_bitwise():
    build.build()
    cases = [problem(260, 280, BC[0], seed=1), problem(261, 281, BC[1], axisym=1, seed=2),
             problem(130, 561, BC[2], seed=3, ch_advection=1), problem(300, 250, BC[2], axisym=1, seed=4),
             problem(33, 17, BC[3], seed=5)]
    tiles = sum(-(-p["nx"] // 26) * -(-p["ny"] // 28) for p, _ in cases)
    assert tiles >= 304
    with gpe2p.Batch([p for p, _ in cases]) as b:
        b.fault(gpe2p.FAULT_FORCE_PERSISTENT, 0)
        for k, (_, f) in enumerate(cases):
            b.init_instance(k, f)
        b.advance(3)
        got = [b.read_instance(k) for k in range(len(cases))]
    for k, (prm, f) in enumerate(cases):
        with gpe2p.Solver(prm) as s:
            s.set_phi_accumulation(gpe2p.PHI_ACC_FP32)
            s.init_fields(f)
            s.advance(3)
            ref = s.read_fields()
        for key in got[k]:
            assert np.array_equal(got[k][key], ref[key]), (k, key)
