"""The 2D FP32 operator check runs the code that steps: the flow step rebuilt from
gpe2p_eval_rates, three stages of TVD-RK3 with phi and mu as given, is the step the
solver takes, bit for bit, at both tile heights, every mix of walls and in the
axisymmetric form.  (The sums of a stage, q + dt L and a q0 + b (q + dt L), are each one
fused multiply-add, formed here exactly and rounded once.)"""
from __future__ import annotations

import numpy as np
import pytest

from paper_2011_00814_gb300 import build, gpe2p, inputs

pytestmark = pytest.mark.gpu

BC = [("periodic", "periodic"), ("noslip", "freeslip"), ("periodic", "noslip"), ("freeslip", "periodic")]
F = np.float32


def fma(a, b, c):
    """a b + c rounded once to FP32: the FP64 sum rounded to odd, then to FP32."""
    p = np.float64(a) * np.float64(b)
    c = np.float64(c)
    s = p + c
    t = s - p
    e = (p - (s - t)) + (c - t)
    even = (s.view(np.int64) & 1) == 0
    return np.where((e != 0) & even, np.nextafter(s, np.where(e > 0, np.inf, -np.inf)), s).astype(F)


@pytest.mark.parametrize("bc", BC)
@pytest.mark.parametrize("size", [(1, 1), (5, 40), (27, 13), (64, 10), (130, 33), (420, 1000)])
def test_flow_step_is_three_stages_of_the_rates(size, bc):
    build.build()
    for axisym in (0, 1):
        if axisym and bc[0] == "periodic":
            continue
        prm = inputs.base_params(2, *size, dx=0.5, dt=0.02, cs=1.2, rhoL=1.0, rhoG=0.3, etaL=0.05, etaG=0.01,
                                 rho_ref=0.6, sigma=0.03, M=0.02, W=2.0, g=(0.0 if axisym else 0.01, -0.02, 0.0),
                                 bc=bc + ("periodic",))
        prm.update(precision=32, axisym=axisym)
        f = {k: v.astype(F).astype(np.float64) for k, v in inputs.random_fields(prm, seed=4).items()}
        dt = F(prm["dt"])
        with gpe2p.Solver(prm) as s:
            s.set_phi_accumulation(gpe2p.PHI_ACC_FP32)
            s.init_fields(f)
            q0 = s.read_fields()
            s.step()
            got = s.read_fields()
            q = q0
            for a, b in ((None, None), (F(0.75), F(0.25)), (F(1.0 / 3.0), F(2.0 / 3.0))):
                s.init_fields(dict(q, phi=f["phi"]))
                L = s.eval_rates()
                n = {}
                for k, r in (("p", "Lp"), ("u", "Lu"), ("v", "Lv")):
                    v = fma(dt, L[r], q[k])
                    if a is not None:
                        v = fma(a, q0[k], F(b) * v)
                    n[k] = v.astype(np.float64)
                q = n
        for k in ("p", "u", "v"):
            assert np.array_equal(q[k], got[k]), (axisym, k)
