"""Diagnostics of batches: the values of one instance and of the whole batch, whatever
the number of blocks an instance is given, and a large instance at the speed of a
single problem."""
from __future__ import annotations

import time

import numpy as np
import pytest

import oracle
from paper_2011_00814_gb300 import build, gpe2p, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    gpe2p.lib()


def problem(nx, ny, seed, precision):
    prm = inputs.base_params(2, nx, ny, dx=0.5, dt=0.02, cs=1.2, rhoL=1.0, rhoG=0.25, etaL=0.05, etaG=0.01, rho_ref=0.6,
                             sigma=0.03, M=0.02, W=2.0, g=(0.0, -0.02, 0.0), bc=("periodic", "noslip", "periodic"))
    prm["precision"] = precision
    return prm, inputs.random_fields(prm, seed=seed)


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("n", [1, 3, 37, 38, 39, 50])     # 1216 blocks over n instances: 32 or fewer from 38 on
def test_batch_diagnostics_match_the_oracle(n, precision):
    sizes = [(1, 1), (5, 3), (300, 2), (64, 64), (2, 700), (257, 40)]
    cases = [problem(*sizes[(k + n) % len(sizes)], seed=k, precision=precision) for k in range(n)]
    with gpe2p.Batch([p for p, _ in cases]) as b:
        for k, (_, f) in enumerate(cases):
            b.init_instance(k, f)
        one = [b.diagnostics(k) for k in range(n)]
        every = b.diagnostics()
        got = [b.read_instance(k) for k in range(n)]
    total = np.zeros(3)
    for k, (p, _) in enumerate(cases):
        ref = oracle.diag(p, got[k])                      # of the stored fields
        cells = p["nx"] * p["ny"] * p["dx"] ** 2
        # FP64 sums of at most 10,280 cells of size one: their rounding is below 1e-12 of
        # the volume
        assert abs(one[k]["int_phi"] - ref[0]) <= 1e-12 * cells
        assert abs(one[k]["kinetic"] - ref[1]) <= 1e-12 * max(ref[1], cells)
        assert abs(one[k]["umax"] - ref[2]) <= 1e-15
        total += (ref[0], ref[1], 0.0)
        total[2] = max(total[2], ref[2])
    volume = sum(p["nx"] * p["ny"] * p["dx"] ** 2 for p, _ in cases)
    assert abs(every["int_phi"] - total[0]) <= 1e-12 * volume
    assert abs(every["kinetic"] - total[1]) <= 1e-12 * volume
    assert abs(every["umax"] - total[2]) <= 1e-15


def test_a_large_instance_is_reduced_by_the_whole_chip():
    """The reduction is bound by the FP64 operations of the SMs that take part: on a
    fifth of them it takes nearly five times as long as a single problem's."""
    prm, _ = problem(4096, 4096, 0, 32)
    f = {k: np.zeros((4096, 4096)) for k in ("phi", "u", "v", "p")}

    def best(diag):
        diag()
        t = []
        for _ in range(10):
            t0 = time.perf_counter()
            diag()
            t.append(time.perf_counter() - t0)
        return min(t)

    with gpe2p.Solver(prm) as s:
        s.init_fields(f)
        alone = best(s.diagnostics)
    with gpe2p.Batch([prm]) as b:
        b.init_instance(0, f)
        batch = best(lambda: b.diagnostics(0))
    print(f"single problem {alone * 1e6:.0f} us, batch of one {batch * 1e6:.0f} us")
    assert batch < 2.0 * alone
