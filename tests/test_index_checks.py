"""The index-checking build tests every population store of the reverse step:
each statement of its source that writes the adjoint populations does so
behind in_bounds.  No GPU is needed."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0803_2826_gb300", "csrc")


def _body(src, name):
    at = src.index(name + "(")
    start = src.index("{", at)
    depth = 0
    for k in range(start, len(src)):
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        if depth == 0:
            return src[start:k]
    raise AssertionError(name)


@pytest.mark.parametrize("function", ["void push_pair", "k_adjoint_step"])
def test_adjoint_stores_are_checked(function):
    body = re.sub(r"//.*", "", _body(open(os.path.join(CSRC, "adjoint.cu")).read(), function))
    # names that stand for lam_out: the argument and pointers made from it
    names = {"lam_out"} | set(re.findall(r"float \*(\w+) = lam_out", body))
    stores = [st for st in body.replace("{", ";").replace("}", ";").split(";")
              if re.search(r"\b(%s)\[[^\]]*\](\])?\s*=[^=]" % "|".join(names), st) or re.search(r"store\((%s)\b" % "|".join(names), st)]
    assert stores
    for st in stores:
        assert "in_bounds(" in st, st.strip()
