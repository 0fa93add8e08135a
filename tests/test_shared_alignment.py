"""Shared arrays that are reached by their 32-bit shared address (inline-PTX vector stores, also from the
other CTAs of a cluster) state the stores' alignment: a complex value is stored by one 8- or 16-byte
instruction, while the value types themselves are only aligned to their parts.  CPU only: the sources
are read."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1706_07919_gb300", "csrc")


def _declarations(src):
    """name -> texts of its static shared declarations"""
    out = {}
    for m in re.finditer(r"^\s*(?!extern)__shared__\s+([^;]+);", src, flags=re.M):
        for name in re.findall(r"(\w+)\s*\[", m.group(1)):
            out.setdefault(name, []).append(m.group(1))
    return out


def test_addressed_shared_arrays_are_aligned():
    checked = set()
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        shared = _declarations(src)
        aligned = set(re.findall(r"struct\s+alignas\(\d+\)\s+(\w+)", src))
        for name in set(re.findall(r"__cvta_generic_to_shared\(&?(\w+)", src)) & set(shared):
            for decl in shared[name]:
                kind = re.match(r"(\w+)", decl).group(1)
                assert decl.startswith("alignas(16)") or kind in aligned, (os.path.basename(path), name, decl)
            checked.add(name)
    assert {"rec", "drow", "xb"} <= checked
