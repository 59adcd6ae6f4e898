"""The autotuner's result file: a line counts only for the table of kernel shapes it was written with.

A shape is an index into that table, which differs between the mechanism structures and has changed
over time, so a line without the table's mark (the form of earlier files) and a line of the other
structure are passed over and the batch is tuned anew.
"""
import numpy as np
import pytest

from chem_inputs import mechanism as M
from chem_inputs import workloads as W
from tests._gpu import to_dev

pytestmark = pytest.mark.gpu


def _tune(species, cache):
    import torch
    from paper_2506_02602_gb300 import build, chem
    build.build()
    ctx = chem.Context(M.build(0) if species == 9 else M.build13(0), "mixed")
    r = W.reactors(96, seed=59) if species == 9 else W.reactors13(96, seed=59)
    Y, T = to_dev(r["Y"]), to_dev(r["T"])
    rho, e = ctx.state_from_TPY(T, to_dev(r["p"]), Y)
    best, table = ctx.autotune_batched(
        rho, e, Y, T, to_dev([0, 32, 96], torch.int64), to_dev([1e-9, 1e-9]), to_dev([1, 2], torch.int32),
        cache_path=str(cache))
    ctx.close()
    return best, table


def test_line_of_an_earlier_form_is_passed_over(tmp_path):
    import torch
    p = torch.cuda.get_device_properties(0)
    cache = tmp_path / "tune.txt"
    old = "%s %d 1 100000 %.6e %.6e 6 1 | 1 1 0 5\n" % (p.name.replace(" ", "_"), p.multi_processor_count, 1e-6, 1e-10)
    cache.write_text(old)
    best, table = _tune(9, cache)
    assert table
    lines = cache.read_text().splitlines(True)
    assert lines[0] == old and len(lines) == 2
    again, table = _tune(9, cache)
    assert not table and again == best


def test_structures_do_not_share_lines(tmp_path):
    cache = tmp_path / "tune.txt"
    assert _tune(9, cache)[1]
    assert _tune(13, cache)[1]
    assert len(cache.read_text().splitlines()) == 2
    assert not _tune(9, cache)[1] and not _tune(13, cache)[1]
