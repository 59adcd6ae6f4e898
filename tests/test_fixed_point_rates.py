"""The fp64 right-hand side's fixed-point exponentials at the edges of their range.

They serve temperatures in (128, 8192) K and coefficients that fit their fixed-point forms; any
other evaluation takes the floating-point exponentials.  Cells on both sides of 128 K, and a
mechanism with one coefficient beyond the forms' range (a temperature exponent of 8, its A
scaled to the same rate at 1500 K), meet the oracle at the same bar as every fp64 cell: 1e-8
relative on T, 1e-10 absolute on Y, equal step counts.
"""
import copy

import numpy as np
import pytest

import oracle
from chem_inputs import mechanism as M
from chem_inputs import workloads as W
from tests._gpu import compare, run_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("species", [9, 13])
@pytest.mark.parametrize("case", ["cold", "wide_exponent", "negative_exponent", "large_energy"])
@pytest.mark.parametrize("n", [1, 257])
def test_edges_of_the_fixed_point_forms(species, case, n):
    from paper_2506_02602_gb300 import build, chem
    build.build()
    mech = copy.deepcopy(M.build(0) if species == 9 else M.build13(0))
    j = 0  # H + O2 = O + OH
    if case == "wide_exponent":
        mech["A"][j] /= 1500.0 ** (8.0 - mech["b"][j])
        mech["b"][j] = 8.0
    elif case == "negative_exponent":
        mech["A"][j] *= 1500.0 ** (7.0 + mech["b"][j])
        mech["b"][j] = -7.0
    elif case == "large_energy":  # Ta = 1e5 K, beyond Ta / ln2 < 130,000 K
        mech["Ea"][4] = 1e5 * 8.31446261815324
    r = W.reactors(n, seed=41) if species == 9 else W.reactors13(n, seed=41)
    if case == "cold":
        r["T"] = np.linspace(110.0, 150.0, n) if n > 1 else np.array([128.0])
    o = oracle.Oracle(mech)
    rho, e = o.state_from_TPY(r["T"], r["p"], r["Y"])
    ref = o.integrate(rho, e, r["Y"], r["T"], 1e-7)
    ctx = chem.Context(mech, "fp64")
    gpu = run_device(ctx, rho, e, r["Y"], r["T"], 1e-7)
    ctx.close()
    compare(gpu, ref)
