"""surrogate_train with epochs 0: the library's default number of epochs, and as many losses."""
import numpy as np
import pytest

from tests import test_surrogate_training as TT

pytestmark = pytest.mark.gpu


def test_zero_epochs_are_the_default():
    from paper_2506_02602_gb300 import build, chem
    build.build()
    n = TT.B + 5
    T, p, Y0, Y1, dt = (TT.to_dev(a) for a in TT._pairs(n))
    ctx = chem.Context(TT.MECH, "fp64")
    rho, e = ctx.state_from_TPY(T, p, Y0)
    loss = {k: ctx.surrogate_train(rho, e, Y0, dt, Y1, T0=T, epochs=k, batch=TT.B, seed=TT.SEED)
            for k in (0, chem.TRAIN_EPOCHS)}
    ctx.close()
    assert loss[0].size == chem.TRAIN_EPOCHS == 20
    np.testing.assert_allclose(loss[0], loss[chem.TRAIN_EPOCHS], rtol=1e-5)
