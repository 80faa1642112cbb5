"""The fused 2D FP32 step at the sizes where its tiles can go wrong: grids
narrower than a tile's halo, one tile, a column or row past a tile edge, both tile
heights, every mix of walls, the axisymmetric form, the compensated phi
accumulation, and more steps than one graph of many steps holds.

Two references.  (1) The FP64 oracle: FP32 rounding of q + dt L is 2^-24 of the
field per stage, so after n steps the relative error of p, u, v, phi stays below
2^-24 x (3 stages + 2 stages) n x 8 (eight: sums of up to a dozen terms each),
which for n = 4 is 1e-5; phi's rounding enters mu through kappa lap ~ 16 kappa /
dx^2, which scales its bound.  (2) The same problem as an instance of a batch in
the persistent form (other tiles), which must give the same bits."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2011_00814_gb300 import build, gpe2p, inputs

pytestmark = pytest.mark.gpu

BC = [("periodic", "periodic"), ("noslip", "freeslip"), ("periodic", "noslip"), ("freeslip", "periodic")]
SIZES = [(1, 1), (2, 3), (5, 40), (26, 12), (27, 13), (25, 29), (64, 10), (53, 57), (130, 33)]
TALL = [(1200, 300), (420, 1000)]


def problem(nx, ny, bc, axisym=0, seed=3):
    prm = inputs.base_params(2, nx, ny, dx=0.5, dt=0.02, cs=1.2, rhoL=1.0, rhoG=0.3, etaL=0.05, etaG=0.01,
                             rho_ref=0.6, sigma=0.03, M=0.02, W=2.0, g=(0.0 if axisym else 0.01, -0.02, 0.0),
                             bc=bc + ("periodic",))
    prm.update(precision=32, axisym=axisym)
    f = inputs.random_fields(prm, seed=seed)
    return prm, {k: v.astype(np.float32).astype(np.float64) for k, v in f.items()}


def run(prm, f, n, mode=gpe2p.PHI_ACC_FP32):
    with gpe2p.Solver(prm) as s:
        s.set_phi_accumulation(mode)
        s.init_fields(f)
        s.advance(n)
        return s.read_fields()


def check(got, ref, tol):
    for k in ("phi", "u", "v", "p"):
        scale = max(np.max(np.abs(ref[k])), 1e-2)
        assert np.max(np.abs(got[k] - ref[k])) <= tol * scale, k
    assert np.max(np.abs(got["mu"] - ref["mu"])) <= tol * 16.0 * 0.75 / 0.25, "mu"


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    gpe2p.lib()


@pytest.mark.parametrize("mode", [gpe2p.PHI_ACC_FP32, gpe2p.PHI_ACC_COMPENSATED])
@pytest.mark.parametrize("bc", BC)
@pytest.mark.parametrize("size", SIZES)
def test_short_tiles_match_oracle_and_batch(size, bc, mode):
    n = 4
    cases = [problem(*size, bc)]
    if bc[0] != "periodic":
        cases.append(problem(*size, bc, axisym=1))
    for prm, f in cases:
        got = run(prm, f, n, mode)
        st = oracle.init_state(prm, f["phi"], f["p"], f["u"], f["v"])
        check(got, oracle.step(prm, st, n), 1e-5)
        if mode == gpe2p.PHI_ACC_FP32:
            with gpe2p.Batch([prm]) as b:
                b.fault(gpe2p.FAULT_FORCE_PERSISTENT, 1)
                b.init_instance(0, f)
                b.advance(n)
                other = b.read_instance(0)
            for k in other:
                assert np.array_equal(got[k], other[k]), k


@pytest.mark.parametrize("size", TALL)
def test_tall_tiles_match_oracle_and_batch(size):
    prm, f = problem(*size, ("noslip", "periodic"))
    got = run(prm, f, 2)
    st = oracle.init_state(prm, f["phi"], f["p"], f["u"], f["v"])
    check(got, oracle.step(prm, st, 2), 1e-5)
    with gpe2p.Batch([prm]) as b:
        b.fault(gpe2p.FAULT_FORCE_PERSISTENT, 1)
        b.init_instance(0, f)
        b.advance(2)
        other = b.read_instance(0)
    for k in other:
        assert np.array_equal(got[k], other[k]), k


@pytest.mark.parametrize("first", [0, 1, 5])
def test_many_steps_in_one_graph(first):
    """advance(n) replays graphs of several steps; the fields, the counter and
    the checks are those of single steps, from either buffer parity."""
    prm, f = problem(60, 40, BC[0])
    with gpe2p.Solver(dict(prm, diag_every=37)) as a, gpe2p.Solver(prm) as b:
        for s in (a, b):
            s.init_fields(f)
            for _ in range(first):
                s.step()
        d = a.advance(75)
        for _ in range(75):
            b.step()
        e = b.diagnostics()
        # the automatic accumulation may switch at the check in the middle: compare before it
        assert d["step"] == e["step"] == first + 75
    with gpe2p.Solver(prm) as a, gpe2p.Solver(prm) as b:
        for s in (a, b):
            s.set_phi_accumulation(gpe2p.PHI_ACC_FP32)
            s.init_fields(f)
            for _ in range(first):
                s.step()
        a.advance(75)
        for _ in range(75):
            b.step()
        x, y = a.read_fields(), b.read_fields()
        for k in x:
            assert np.array_equal(x[k], y[k]), k
