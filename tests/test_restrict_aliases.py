"""The kernels' __restrict__ pointers never name one array twice: within a
function, an array of the context (p.F, p.A4, ...) that a __restrict__ pointer
to non-const may write is behind no other __restrict__ pointer in the same
stage.  (The compiler may assume so, and read such an array early or through
the read-only cache.)"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1909_08390_gb300", "csrc")
STAGES = ("kPrep", "kStage3", "kStage4", "kFinal")
DECL = re.compile(r"(const )?(?:double|float)\* __restrict__ (?:const )?(\w+) =\s*([^;]*);")


def array_of(expr, stage):
    """The array that a chain of STAGE comparisons picks for a stage."""
    expr = re.sub(r"\((?:const )?(?:double|float)\*\)", "", expr).replace("(", " ").replace(")", " ")
    while "?" in expr:
        cond, rest = expr.split("?", 1)
        yes, no = rest.split(":", 1)
        expr = yes if re.search(r"STAGE == (\w+)", cond).group(1) == stage else no
    m = re.search(r"\bp\.(\w+)", expr)
    return m.group(1) if m else None


@pytest.mark.parametrize("name", ["fdlb_kernels.cu", "fdlb_mixed.cu", "fdlb_adjoint.cu"])
def test_restrict_pointers_do_not_alias(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    found = 0
    for body in re.split(r"\n}\n", text):  # functions end at column 0
        decls = [(bool(c), var, init) for c, var, init in DECL.findall(body)]
        found += len(decls)
        for stage in STAGES:
            held = [(const, var, array_of(init, stage)) for const, var, init in decls]
            for i, (const, var, array) in enumerate(held):
                for other_const, other, other_array in held[i + 1:]:
                    if array and array == other_array:
                        assert const and other_const, (name, stage, var, other, array)
    assert found or name == "fdlb_adjoint.cu"
