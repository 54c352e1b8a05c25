"""Multipliers are loaded without the read-only path.

The persistent kernels rewrite y and y~ while they run, and read them after other blocks
wrote them.  `ld.global.nc` (`__ldg`) is undefined for such data: a line cached in an
earlier iteration may come back.  The bodies of these kernels load both through
ld_multiplier.
"""
import re
from pathlib import Path

import pytest

import paper_2407_15049_gb300 as L

CSRC = Path(L.__file__).resolve().parent / "csrc"
# loads of y, y~ (y, ydf, ytil; v of the product over the constraints' pattern) by the read-only path
READ_ONLY = re.compile(r"(__ldg\((static_cast<[^>]*>\()?(y|ydf|ytil)\b|ld_scalar<\w+>\((y|nullptr), (ydf|static_cast<const dfloat\*>\(v\)))")


@pytest.mark.parametrize("name", ["kernels.cuh", "cons.cuh", "admm.cuh", "batch_kernel.cuh"])
def test_persistent_bodies_load_multipliers_plainly(name):
    assert not READ_ONLY.findall((CSRC / name).read_text())


def test_pattern_weight_loads_the_multiplier_plainly():
    text = (CSRC / "kernels.cuh").read_text()
    at = text.index("spmm_a_weight(")
    body = text[at:text.index("\n}", at)]
    assert not re.search(r"__ldg\(static_cast<const double\*>\(v\)", body)
    assert "ld_multiplier" in body
