"""The mixed variant's double-float temperature solve at the edges of its range.

Its Newton iteration keeps to the NASA-7 range of its starting guess and leaves the rest to the
fp64 solve: guesses that are missing, of the wrong sign or far off, roots on the other side of
the range switch, and cells whose temperature crosses it within the step.  Each such cell has to
come out as from any other guess: the mixed bar (1e-5 relative on T) against the oracle started
from the same guess, and T solved from the final state to |dT| <= 1e-12 T (so e(T, Y) meets e to
about c_v 1e-12 T, 1e-5 J/kg).  129 cells: one more than a block of the default shape.
"""
import numpy as np
import pytest

import oracle
from chem_inputs import mechanism as M
from chem_inputs import workloads as W
from tests._gpu import run_device

pytestmark = pytest.mark.gpu

N = 129


def _case(species):
    mech = M.build(0) if species == 9 else M.build13(0)
    r = W.reactors(N, seed=31) if species == 9 else W.reactors13(N, seed=31)
    o = oracle.Oracle(mech)
    r["T"][:60] = 1000.0 + np.linspace(-0.3, 0.3, 60)  # around the NASA-7 switch at 1000 K
    return mech, o, r


@pytest.mark.parametrize("species", [9, 13])
@pytest.mark.parametrize("guess", ["given", "nan", "zero", "negative", "cold", "hot", "far"])
def test_guesses_and_range_switch(species, guess):
    from paper_2506_02602_gb300 import build, chem
    build.build()
    mech, o, r = _case(species)
    rho, e = o.state_from_TPY(r["T"], r["p"], r["Y"])
    T = r["T"].copy()
    if guess != "given":
        T[:] = {"nan": np.nan, "zero": 0.0, "negative": -5.0, "cold": 300.0, "hot": 4000.0, "far": 5e4}[guess]
    ref = o.integrate(rho, e, r["Y"], T, 1e-6)
    ctx = chem.Context(mech, "mixed")
    gpu = run_device(ctx, rho, e, r["Y"], T, 1e-6)
    ctx.close()
    np.testing.assert_array_equal(gpu["status"], ref["status"])
    ok = ref["status"] == 0  # from 5e4 K the extrapolated polynomials lead some cells nowhere
    assert ok.any() or guess == "far"
    assert np.max(np.abs(gpu["T"] - ref["T"])[ok] / ref["T"][ok], initial=0.0) <= 1e-5
    assert np.max(np.abs(gpu["Y"] - ref["Y"])[:, ok], initial=0.0) <= 1e-6
    e_out = np.array([o.e_mix(gpu["Y"][:, i], gpu["T"][i]) for i in np.flatnonzero(ok)])
    np.testing.assert_allclose(e_out.reshape(-1), e[ok], rtol=1e-12, atol=1e-5)
