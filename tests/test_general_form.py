"""The fp64 right-hand side's general form is compiled into the kernels (ptxas reports of the in-tree
build, on the CPU): as a function of its own it reads every coefficient through memory and takes two
to three times as long, which is what a mechanism outside the fixed-point tables' ranges then pays on
each evaluation."""
import os

import pytest

from paper_2506_02602_gb300 import build


@pytest.mark.parametrize("lib", sorted(build.LIBS))
def test_general_form_is_inlined(lib):
    build.build()
    reports = [os.path.join(build.LIBS[lib]["build"], u + ".ptxas.txt") for u in ("integrate", "batched")]
    for path in reports:
        with open(path) as f:
            text = f.read()
        assert "k_lsrk" in text
        assert "cell_rhs_any" not in text, path
