"""The temperature of the fp64 kernel's fixed-point solve against the root in extended precision (numpy's
longdouble: 64 bits of mantissa or more).

Tolerance: the last step (at most 4e-9 T) is off by its fp32 slope's 2^-20, T is rounded to fp64, the
residual is off by 32 units of 2^-33 of e/R_u and e/R_u itself rounded.  The second test's is what fp64
sums leave: the rounding of T and 8 roundings of the largest term of e/R_u.
"""
import numpy as np
import pytest

import oracle
from chem_inputs import mechanism as M
from chem_inputs import workloads as W
from tests._gpu import run_device

pytestmark = pytest.mark.gpu

L = np.longdouble
RU = 8.31446261815324


def _solved(species, Y, T, p, guess):
    """(T of cells advanced by 1e-30 s, so that their composition does not change, its error, c_v / R_u, e / R_u,
    the largest term of e / R_u)"""
    from paper_2506_02602_gb300 import build, chem
    build.build()
    mech = M.build(0) if species == 9 else M.build13(0)
    rho, e = oracle.Oracle(mech).state_from_TPY(T, p, Y)
    ctx = chem.Context(mech, "fp64")
    gpu = run_device(ctx, rho, e, Y, guess, 1e-30)
    ctx.close()
    assert np.all(gpu["status"] == 0)
    assert np.max(np.abs(gpu["Y"] - Y)) < 1e-18
    # the root of e(T) = e by Newton in extended precision
    a = [np.array(mech[k], dtype=np.float64).astype(L) for k in ("nasa_lo", "nasa_hi")]
    W_ = np.array(mech["W"], dtype=np.float64).astype(L)
    yw, eR, Tm = Y.astype(L) / W_[:, None], e.astype(L) / L(RU), float(mech["T_mid"][0])
    mix = [np.stack([(c[:, i] * yw.T).sum(1) for i in range(6)]) for c in a]
    t = gpu["T"].astype(L)
    for _ in range(4):
        m = np.where(t >= Tm, mix[1], mix[0])
        cv = m[0] - yw.sum(0) + t * (m[1] + t * (m[2] + t * (m[3] + t * m[4])))
        terms = [t * (m[0] - yw.sum(0))] + [t ** (i + 1) * m[i] / (i + 1) for i in range(1, 5)] + [m[5]]
        t = t - (sum(terms) - eR) / cv
    err = np.abs(gpu["T"].astype(L) - t)
    print(f"\nT: {float((err / t).max()):.3g} relative")
    return t, err, cv, np.abs(eR), np.max(np.abs(np.stack(terms)), axis=0)


@pytest.mark.parametrize("species", [9, 13])
def test_temperature(species):
    """Random compositions over (140, 8000) K and around the NASA-7 ranges' common temperature, from guesses
    0 to 30 % off."""
    n = 4096
    r = W.reactors(n, seed=61) if species == 9 else W.reactors13(n, seed=61)
    rng = np.random.default_rng(61)
    Y = 0.7 * r["Y"] + 0.3 * rng.dirichlet(np.ones(species), n).T
    T = np.concatenate([np.exp(rng.uniform(np.log(140.0), np.log(8000.0), n - 512)), np.linspace(999.99, 1000.01, 512)])
    guess = np.clip(T * rng.choice([1.0, 1.0 + 1e-9, 1.001, 1.3, 0.77], n), 130.0, 8100.0)
    t, err, cv, eR, _ = _solved(species, Y, T, r["p"], guess)
    assert np.all(err <= (4e-9 * 2.0**-20 + 2.0**-52) * t + 32 * 2.0**-33 / cv + eR * 2.0**-52 / cv)


@pytest.mark.parametrize("species", [9, 13])
@pytest.mark.parametrize("state", ["reactors", "slice", "cold"])
def test_temperature_is_as_exact_as_fp64(species, state):
    """The workloads' own states."""
    n = 4096
    if state == "slice":
        r = W.detonation_slice(64, 64) if species == 9 else W.detonation_slice13(64, 64)
    else:
        r = W.reactors(n, seed=67) if species == 9 else W.reactors13(n, seed=67)
    T = np.linspace(280.0, 330.0, n) if state == "cold" else r["T"]
    rng = np.random.default_rng(67)
    guess = T * rng.choice([1.0, 1.0 - 1e-7, 1.001, 1.2, 0.9], n)
    t, err, cv, eR, term = _solved(species, r["Y"], T, r["p"], guess)
    assert np.all(err <= 2.0**-52 * t + 8 * 2.0**-53 * np.maximum(eR, term) / cv)
