"""The training pass's weight and bias gradients at the edges of the GEMM's row and K tiles.

The batch is the K of the weight gradients, split over 16 slices and staged 256 at a time: one
row, a partial last slice, K tails off the 8- and 64-row grids and more than one staged group per
slice (16 x 256 rows and beyond).  Each gradient is compared with the fp64 product of the pass's own
bf16 factors; fp32 sums of B terms in any order are within (B + 16) 2^-23 of sum |terms|.
"""
import numpy as np
import pytest

from tests import test_surrogate as TS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 65, 1023, 4096, 4099, 20001])
def test_gradients_at_ragged_batches(B):
    from paper_2506_02602_gb300 import build, chem
    build.build()
    ctx = chem.Context(TS.MECH, "fp64")
    TS._bf16_network(ctx)
    Xb, Tt = TS._batch(B)
    tr = ctx.surrogate_trace(Xb.cuda(), Tt.cuda())
    grads = TS._from_gpu_layout(tr["grad"].astype(np.float64))
    ctx.close()
    H = [Xb.numpy().astype(np.float64)] + [tr["H"][l].astype(np.float64) for l in range(3)]
    G = [tr["G"][l].astype(np.float64) for l in range(3)] + [tr["G3"].astype(np.float64)]
    eps = (B + 16) * 2.0 ** -23
    for l in range(4):
        W, b = grads[l]
        assert np.all(np.abs(W - G[l].T @ H[l]) <= eps * (np.abs(G[l]).T @ np.abs(H[l])) + 1e-30), l
        assert np.all(np.abs(b - G[l].sum(0)) <= eps * np.abs(G[l]).sum(0) + 1e-30), l
