"""chem_surrogate_train step by step: its captured steps (gather by the step counter, weight gradients on a
second stream, Adam with the schedule's entry of the step and the split sums) against the same steps
through chem_surrogate_grad and chem_surrogate_adam, with the permutations, features and learning rates
restated here.

The number of batches goes around the eight steps of a replayed graph, over two epochs, with rows left over.
Both sides run the same GEMMs, so what differs are features that a last-bit difference of log or pow
takes across a bf16 rounding (a relative 2^-8 of one input, rarely): far below 2 % of a parameter's path
(the sum of the learning rates) for 99 of 100 parameters, and a wrong batch, schedule entry or slice
moves nearly all of them by more than that.  A parameter whose gradient is all but zero may go either way,
twice the path at most.
"""
import struct

import numpy as np
import pytest

from chem_inputs import mechanism as M
from chem_inputs import workloads as W
from tests._gpu import to_dev

pytestmark = pytest.mark.gpu

MECH = M.build(0)
B, EPOCHS, SEED, LR, LR_END, LAM = 96, 2, 5, 1e-3, 1e-4, 0.1
M64 = 2**64 - 1


def _pairs(n):
    r = W.reactors(n, seed=71)
    rng = np.random.default_rng(71)
    Y0 = 0.9 * r["Y"] + 0.1 * rng.dirichlet(np.ones(9), n).T
    Y1 = Y0 * np.exp(0.2 * rng.standard_normal(Y0.shape))
    dt = np.exp(rng.uniform(np.log(1e-9), np.log(1e-7), n))
    return r["T"], r["p"], Y0, Y1 / Y1.sum(0), dt


def _permutations(n):
    state = SEED ^ 0x5BD1E995
    while True:
        perm = list(range(n))
        for i in range(n - 1, 0, -1):
            state = (state + 0x9E3779B97F4A7C15) & M64
            z = state
            z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
            j = (z ^ (z >> 31)) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        yield np.array(perm)


def _boxcox(Y):
    return (np.maximum(Y, 1e-30) ** LAM - 1) / LAM


@pytest.mark.parametrize("nb", [1, 7, 8, 9, 16])
def test_training_is_the_sum_of_its_steps(nb, tmp_path):
    import torch
    from paper_2506_02602_gb300 import build, chem
    build.build()
    n = nb * B + 13
    T, p, Y0, Y1, dt = _pairs(n)
    ctx = chem.Context(MECH, "fp64")
    d = [to_dev(a) for a in (T, p, Y0, Y1, dt)]
    rho, e = ctx.state_from_TPY(d[0], d[1], d[2])
    train = lambda epochs, lr: ctx.surrogate_train(rho, e, d[2], d[4], d[3], T0=d[0], epochs=epochs, batch=B, lr=lr,  # noqa: E731
                                                   lr_final=LR_END / LR * lr, boxcox_lambda=LAM, seed=SEED)
    train(1, 1e-30)  # steps of 1e-30 leave the initial parameters as they are
    start = ctx.surrogate_params()
    loss = train(EPOCHS, LR)
    got = ctx.surrogate_params()
    path = tmp_path / "net.bin"
    ctx.surrogate_save(str(path))
    norm = np.frombuffer(path.read_bytes()[8 + struct.calcsize("<qdd"):][: 88 * 4], np.float32)
    fmean, fistd, _, _, tmean, tistd = np.split(norm, [16, 32, 44, 56, 72])
    X = np.zeros((n, 16), np.float32)
    D = np.zeros((n, 16), np.float32)
    X[:, :12] = np.concatenate([np.stack([T, np.log(p), np.log10(dt)]), _boxcox(Y0)]).T
    D[:, :9] = (_boxcox(Y1) - _boxcox(Y0)).T
    X, D = (X - fmean) * fistd, (D - tmean) * tistd
    ctx.surrogate_params(start)
    total, step, want_loss, reach = nb * EPOCHS, 0, [], 0.0
    for _, perm in zip(range(EPOCHS), _permutations(n)):
        losses = []
        for b in range(nb):
            rows = perm[b * B:(b + 1) * B]
            _, g, f = ctx.surrogate_grad(torch.tensor(X[rows], device="cuda"), torch.tensor(D[rows], device="cuda"))
            lr = np.float32(LR_END + 0.5 * (LR - LR_END) * (1 + np.cos(np.pi * (step / (total - 1) if total > 1 else 1.0))))
            ctx.surrogate_adam(g, lr)
            losses.append(f)
            reach += float(lr)
            step += 1
        want_loss.append(np.mean(losses))
    want = ctx.surrogate_params()
    ctx.close()
    np.testing.assert_allclose(loss, want_loss, rtol=1e-3)
    assert np.abs(want - start).mean() > 0.1 * reach
    err = np.abs(got - want) / reach
    print(f"\n99 % within {np.quantile(err, 0.99):.2g} of the path, all within {err.max():.2g}")
    assert np.quantile(err, 0.99) <= 0.02 and err.max() <= 2.0
