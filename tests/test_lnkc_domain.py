"""chem_diag_ln_inv_kc outside its domain: every exponent is NaN at temperatures that are not positive
and finite, and what it gives beside them does not change."""
import numpy as np
import pytest

from chem_inputs import mechanism as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("species", [9, 13])
@pytest.mark.parametrize("form", [0, 1])
def test_non_positive_temperatures_give_nan(species, form):
    import torch
    from paper_2506_02602_gb300 import build, chem
    build.build()
    ctx = chem.Context(M.build(0) if species == 9 else M.build13(0), "mixed")
    bad = [-1000.0, -300.0, -1e-3, 0.0, -0.0, np.nan, np.inf, -np.inf]
    T = np.empty(2 * len(bad) + 1)
    T[1::2] = bad
    T[0::2] = np.linspace(300.0, 3000.0, len(bad) + 1)
    f = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    got = ctx.ln_inv_kc(f(T), form=form).cpu().numpy()
    good = ctx.ln_inv_kc(f(T[0::2].copy()), form=form).cpu().numpy()
    ctx.close()
    assert np.isnan(got[1::2]).all()
    assert np.isfinite(good).all()
    np.testing.assert_array_equal(got[0::2], good)
