"""Inline assembly that writes memory says so.  Without the clobber the compiler may take it that nothing writes the array and move or drop the
ordinary loads that read it back; results cannot show that reliably, so the sources are looked at."""
import glob
import os
import re

import pytest

from conftest import ROOT

SOURCES = {os.path.basename(p): open(p).read() for p in sorted(glob.glob(os.path.join(ROOT, "paper_2608_16329_b200", "csrc", "*.cu*")))}
STORES = r"(?<![\w.])(?:st\.(?:shared|global|volatile|release|relaxed|u|b|f|v)|red\.|atom\.|cp\.async\.c|cp\.async\.bulk|tcgen05\.(?:st|alloc|cp)|stmatrix)"


def _statements(text):
    """The asm statements, with the macros of string literals that they use put in."""
    text = re.sub(r"//[^\n]*", "", text)
    macros = dict(re.findall(r'#define (\w+) ((?:[^\n]*\\\n)*[^\n]*)', text))
    for m in re.finditer(r"\basm\b(?:\s+volatile)?\s*\(", text):
        depth, at = 1, m.end()
        quoted = False
        while depth:
            c = text[at]
            if c == '"' and text[at - 1] != "\\":
                quoted = not quoted
            elif not quoted:
                depth += (c == "(") - (c == ")")
            at += 1
        body = text[m.end():at - 1]
        yield re.sub(r"\b[A-Z]\w+\b", lambda w: macros.get(w.group(), w.group()), body)


def test_the_scan_sees_stores():
    found = [s for text in SOURCES.values() for s in _statements(text) if re.search(STORES, s)]
    assert len(found) > 10 and any("st.shared.u16 [at]" in s for s in found) and any("tcgen05.st" in s for s in found)


@pytest.mark.parametrize("name", sorted(SOURCES))
def test_assembly_that_writes_memory_has_the_clobber(name):
    for statement in _statements(SOURCES[name]):
        if re.search(STORES, statement):
            assert re.search(r':\s*"memory"\s*$', statement.strip()), statement
