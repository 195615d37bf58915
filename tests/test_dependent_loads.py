"""A kernel that waits for the launch before it (pdl_wait) can be resident while
that one still writes, so what it reads of the stream's data must not go
through the read-only load path, which holds a value for constant over the
kernel's whole lifetime: only the grid's tables may.  Read off the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(__file__)), "paper_2103_10114_gb300", "csrc")


def _functions():
    """(name, parameters, body) of every function that pdl_wait() appears in."""
    out = []
    for f in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"pdl_wait\(\);", text):
            start = text.rfind("\ntemplate", 0, m.start())
            end = text.find("\n}", m.start())
            decl, body = text[start:end].split("{", 1)
            name = re.findall(r"(\w+)\(", re.sub(r"__launch_bounds__\([^{]*?\)\s", "", decl))[0]
            out.append((name, decl, body))
    assert {n for n, _, _ in out} >= {"k_adj_col", "adj_row", "k_adj_colstate", "k_row_stage", "row_segment"}
    return out


@pytest.mark.parametrize("fn", _functions(), ids=lambda f: f[0])
def test_only_tables_are_read_through_the_read_only_path(fn):
    name, decl, body = fn
    assert "__restrict__" not in decl, name
    for arg in re.findall(r"\b(?:__)?ldg\(\s*([\w.]+)", body):
        assert arg.startswith("g."), (name, arg)
