"""The fp64 right-hand side's fixed-point form at the edges of its arguments' range.

It serves T in (128, 8192) K, |Y_k| < 1.25 and rho in (2^-64, 2^64); other evaluations take the
floating-point form.  Cells on both sides of 8192 K, with a mass fraction beyond 1.25 and with a
density below 2^-64, and cells whose Newton iteration crosses the NASA-7 ranges' common
temperature, meet the oracle at the same bar as every fp64 cell: 1e-8 relative on T, 1e-10
absolute on Y, equal step counts.

Two more lie inside the range where a logarithm leaves (-32, 32): a density of 2^-40, and Troe
temperatures that put F_cent near 2^-70.
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
@pytest.mark.parametrize("case", ["hot", "crossing", "large_fraction", "thin", "thin_inside", "deep_troe"])
@pytest.mark.parametrize("n", [1, 257])
def test_edges_of_the_fixed_point_arguments(species, case, n):
    from paper_2506_02602_gb300 import build, chem
    build.build()
    mech = copy.deepcopy(M.build(0) if species == 9 else M.build13(0))
    r = W.reactors(n, seed=43) if species == 9 else W.reactors13(n, seed=43)
    dt, guess = 1e-7, None
    if case == "hot":
        r["T"] = np.linspace(8150.0, 8230.0, n) if n > 1 else np.array([8192.0])
        dt = 1e-10
    elif case == "crossing":
        r["T"] = np.linspace(999.0, 1001.0, n)
        guess = np.where(np.arange(n) % 2, 1005.0, 995.0)
    elif case == "large_fraction":
        r["Y"] = 2.0 * r["Y"]
    elif case == "deep_troe":  # exp(-T/T***), exp(-T/T*) and exp(-T**/T) of about e^-50
        j = 8  # H + O2 (+M) = HO2 (+M)
        mech["troe"][j] = [0.5, 30.0, 31.0, 8e4]
    o = oracle.Oracle(mech)
    rho, e = o.state_from_TPY(r["T"], r["p"], r["Y"])
    if case.startswith("thin"):
        rho = np.full(n, 2.0 ** (-65 if case == "thin" else -40))
    T0 = r["T"] if guess is None else guess
    ref = o.integrate(rho, e, r["Y"], T0, dt)
    ctx = chem.Context(mech, "fp64")
    gpu = run_device(ctx, rho, e, r["Y"], T0, dt)
    ctx.close()
    compare(gpu, ref)
