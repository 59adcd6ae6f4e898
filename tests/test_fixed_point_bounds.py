"""The fp64 right-hand side's fixed-point Gibbs sums at the bound of their coefficients.

The polynomial part of -g_k / (R_u T ln2) is a 64-bit sum in units of 2^-56, so it has to stay below
128 up to 8192 K.  HO2 gets linear to quartic terms of one sign that add up to `total` at 8192 K, just
inside and beyond that bound, in tables that stay continuous at their common temperature (and the
reactions that consume it are made irreversible, or such a stable molecule would form at e^100 times
the usual rates).  Whichever form serves the cells, they meet the oracle at the bar of every fp64 cell
(1e-8 relative on T, 1e-10 absolute on Y, equal step counts) where the sum is at its largest.
"""
import copy

import numpy as np
import pytest

import oracle
from chem_inputs import mechanism as M
from chem_inputs import workloads as W
from tests._gpu import compare, run_device

pytestmark = pytest.mark.gpu


def _mechanism(species, total):
    mech = copy.deepcopy(M.build(0) if species == 9 else M.build13(0))
    k, S, Tm = 6, 8192.0, float(mech["T_mid"][0])
    lo = np.array(mech["nasa_lo"][k], dtype=np.float64)
    hi = np.zeros(7)
    i = np.arange(1, 5)
    share = np.array([0.3, 0.3, 0.2, 0.2]) * total / 1.4426950408889634  # a_(i+1) S^i / (i (i + 1))
    hi[1:5] = share * i * (i + 1) / S**i
    for c, f in ((0, lambda a: a[0] + (a[1:5] * Tm**i).sum()),                              # cp / R
                 (5, lambda a: a[0] * Tm + (a[1:5] * Tm**(i + 1) / (i + 1)).sum() + a[5]),  # h / R
                 (6, lambda a: a[0] * np.log(Tm) + (a[1:5] * Tm**i / i).sum() + a[6])):     # s / R
        hi[c] += f(lo) - f(hi)
    mech["nasa_hi"] = np.array(mech["nasa_hi"], dtype=np.float64)
    mech["nasa_hi"][k] = hi
    mech["reversible"] = np.where(np.asarray(mech["nu_f"])[:, k] > 0, 0, mech["reversible"])
    return mech


@pytest.mark.parametrize("species", [9, 13])
@pytest.mark.parametrize("total", [126.0, 145.0, 160.0])
def test_gibbs_polynomial_at_its_bound(species, total):
    from paper_2506_02602_gb300 import build, chem
    build.build()
    n = 129
    mech = _mechanism(species, total)
    r = W.reactors(n, seed=53) if species == 9 else W.reactors13(n, seed=53)
    r["T"] = np.linspace(7700.0, 8150.0, n)
    o = oracle.Oracle(mech)
    rho, e = o.state_from_TPY(r["T"], r["p"], r["Y"])
    ref = o.integrate(rho, e, r["Y"], r["T"], 1e-10, max_steps=500)
    assert np.all(ref["status"] == 0)
    ctx = chem.Context(mech, "fp64", max_steps=500)
    gpu = run_device(ctx, rho, e, r["Y"], r["T"], 1e-10)
    ctx.close()
    compare(gpu, ref)
