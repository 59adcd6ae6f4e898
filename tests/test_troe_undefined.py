"""Fall-off reactions whose Troe broadening factor is not a number.

F_cent = (1 - alpha) exp(-T/T***) + alpha exp(-T/T*) + exp(-T**/T) can be negative for alpha outside
[0, 1], infinite for a large negative T** and not a number for such an alpha; log F_cent, the rate and
the right-hand side are then no numbers either, and the cell ends with the oracle's failure status
instead of a state.  "crossing" has F_cent change its sign near 1200 K, in the middle of the reactors'
temperatures; "growing" stays finite (exp(-T**/T) up to e^5).  Cells that succeed meet the bar of every
fp64 cell (1e-8 relative on T, 1e-10 absolute on Y, equal step counts).
"""
import copy

import numpy as np
import pytest

import oracle
from chem_inputs import mechanism as M
from chem_inputs import workloads as W
from tests._gpu import compare, run_device

pytestmark = pytest.mark.gpu

TROE = {"crossing": [1.8, 1e4, 1300.0, 8e4], "negative_alpha": [-0.5, 300.0, 1e4, 8e4],
        "nan_alpha": [np.nan, 300.0, 1e4, 8e4], "overflow": [0.5, 300.0, 1e4, -2e6],
        "growing": [0.5, 300.0, 1e4, -5e3]}


@pytest.mark.parametrize("species", [9, 13])
@pytest.mark.parametrize("case", sorted(TROE))
@pytest.mark.parametrize("params", [3, 4])
def test_status_of_undefined_broadening(species, case, params):
    if params == 3 and case in ("overflow", "growing"):
        pytest.skip("T** belongs to the four-parameter form")
    from paper_2506_02602_gb300 import build, chem
    build.build()
    n = 129
    mech = copy.deepcopy(M.build(0) if species == 9 else M.build13(0))
    j = int(np.flatnonzero((mech["rtype"] == 2) & (mech["troe_n"] == params))[0])
    mech["troe"][j] = TROE[case]
    r = W.reactors(n, seed=47) if species == 9 else W.reactors13(n, seed=47)
    o = oracle.Oracle(mech)
    rho, e = o.state_from_TPY(r["T"], r["p"], r["Y"])
    ref = o.integrate(rho, e, r["Y"], r["T"], 1e-7)
    bad = int((ref["status"] != 0).sum())
    assert (0 < bad < n) if case == "crossing" else bad == (0 if case == "growing" else n)
    ctx = chem.Context(mech, "fp64")
    gpu = run_device(ctx, rho, e, r["Y"], r["T"], 1e-7)
    ctx.close()
    compare(gpu, ref)
