"""Node-node interactions on the independent components (harmonic folding of
moments, derivatives and coefficients) against the oracle's full tensors: every
order, a set far from the origin (the rounding of the centres is then a dipole
of 1e-9, which the FP64 form carries as an offset of the source's centre; the
oracle's centres round otherwise, which moves the truncation error, so there
the total momentum is what is compared: it vanishes to rounding only if the
expansions of the two sides of a pair agree) and lengths beyond the range in which powers
of 1/r are formed directly."""
import numpy as np
import pytest

import oracle
import workloads
from gpu_helpers import TOL_FP32_MAX, TOL_MOM_FP32, TOL_MOM_FP64, acc_rel, momentum_residual, pot_rel, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("what", ["plain", "shifted", "short", "long"])
def test_fold_matches_full_tensors(order, what):
    pos, m, h = workloads.plummer(3000, 40 + order)
    m = m * np.random.default_rng(order).uniform(0.5, 1.5, len(m))
    if what == "shifted":
        pos = pos + np.array([3e6, -1e6, 2e6])
    scale = {"short": 1e-24, "long": 1e24}.get(what, 1.0)
    pos, h = pos * scale, h * scale
    acc_o, pot_o, st_o = oracle.sfmm(pos, m, h, theta=0.6, p=order, leaf_size=8)
    for prec, tol in (("fp64", 1e-12), ("fp32", TOL_FP32_MAX)):
        if prec == "fp32" and scale != 1.0:
            continue  # beyond the FP32 form's range
        tol = max(tol, 1e-8) if what == "shifted" else tol
        for sched in (1, 2, 3):
            s = solver(prec, schedule=sched)
            s.build(pos, m, h, 8)
            acc, pot = (t.cpu().numpy() for t in s.gravity(0.6, order))
            assert s.stats()["m2l_unique"] == st_o["m2l_unique"]
            s.close()
            assert acc_rel(acc, acc_o).max() <= tol, (prec, sched)
            assert pot_rel(pot, pot_o).max() <= tol, (prec, sched)
            assert momentum_residual(m, acc) <= (TOL_MOM_FP64 if prec == "fp64" else TOL_MOM_FP32), (prec, sched)
