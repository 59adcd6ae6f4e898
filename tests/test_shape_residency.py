"""Resident CTAs per SM of the persistent kernel's shapes on the GPU: what registers and shared memory
(per-thread columns and tables) leave of the counts that the registers are capped for."""
import pytest

from chem_inputs import mechanism as M

pytestmark = pytest.mark.gpu

RESIDENT = {("fp64", 9): [3, 2, 3, 5, 5, 2], ("fp64", 13): [2, 2, 2, 4, 4, 1],
            ("mixed", 9): [4, 3, 2, 6, 7, 2], ("mixed", 13): [3, 3, 2, 5, 5, 1]}


@pytest.mark.parametrize("variant,species", sorted(RESIDENT))
def test_resident_ctas(variant, species):
    from paper_2506_02602_gb300 import build, chem
    build.build()
    ctx = chem.Context(M.build(0) if species == 9 else M.build13(0), variant)
    got = [ctx.batch_shape_info(s) for s in range(chem.BATCH_SHAPES)]
    ctx.close()
    assert [g[0] for g in got] == [128, 128, 128, 64, 64, 256]
    assert [g[2] for g in got] == RESIDENT[variant, species]
