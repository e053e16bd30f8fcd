"""Kernel variants at the sizes and values where they can go wrong, against the oracle."""
import numpy as np
import pytest

import workloads as W
from tests._pair import gpu_f, oracle_of, rel_err, solver_of

pytestmark = pytest.mark.gpu


def _lbs():
    import paper_1702_01335_gb300 as P
    return P


@pytest.mark.parametrize("pattern", ["rest", "jump", "spike", "staircase", "ramp", "scales"])
def test_fp64_weno_weights_at_vanishing_indicators(pattern):
    """The FP64 WENO weights where one, two or all three smoothness indicators vanish or
    differ by tens of orders of magnitude, per velocity: constant stretches next to a jump, a
    single-cell spike, a staircase, an exactly linear ramp and cell values from 1e-300 to 1.
    One step from that state; both sides round the same few dozen operations, so 1e-13 of the
    largest population bounds them."""
    P = _lbs()
    p = dict(W.C1, Nz=24)
    o = oracle_of(p, None)
    s = solver_of(p, o.dt, P.LBS_FP64)
    z, k = np.arange(24)[:, None], np.arange(o.Q)[None, :]
    d = {"rest": 0.0 * (z + k),
         "jump": 0.1 * (z >= 7 + k % 9),
         "spike": 0.1 * (z == 3 + k % 17),
         "staircase": 0.01 * ((z + k) // 5),
         "ramp": (z - 12) * 2.0 ** -8 + 0.0 * k,
         "scales": 0.1 * 10.0 ** (-12.5 * ((z + k) % 24))}[pattern]
    d = np.ascontiguousarray(d, dtype=np.float64)
    s.set_state(0, d)
    o.f[3:-3] = (1.0 + d) * o.weights()[None, :]
    s.step(1)
    o.step(1)
    assert rel_err(gpu_f(s, o), o.f[3:3 + o.Nz]) < 1e-13
