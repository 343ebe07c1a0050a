"""Every launch wrapper that the library's internal header declares has a caller, and no wrapper or kernel takes a status
word that it does not use (from the sources, on the CPU)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1111_4363_gb300", "csrc")


def source(name):
    return re.sub(r"//[^\n]*", "", open(name).read())


def test_every_declared_launcher_is_called():
    header = os.path.join(CSRC, "la_internal.cuh")
    names = set(re.findall(r"\b(launch_\w+|norm_blocks|galerkin_table_doubles|encode_\w+)\s*\(", source(header)))
    assert len(names) > 20
    text = "\n".join(source(f) for f in glob.glob(os.path.join(CSRC, "*.cu*")) if f != header) + source(header)
    for n in sorted(names):
        calls = [m for m in re.finditer(rf"\b{n}\b(?:<[^<>;()]*>)?\s*\(", text)
                 if not re.search(r"(?:void|cudaError_t|bool|int|long long)\s+$", text[max(0, m.start() - 30):m.start()])]
        assert calls, n


def test_no_unused_status_parameter():
    text = "\n".join(source(f) for f in glob.glob(os.path.join(CSRC, "*.cu*")))
    for m in re.finditer(r"\b(\w+)\s*\(([^;{}()]*int\*\s*(?:__restrict__\s*)?status\b[^;{}()]*)\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        assert re.search(r"\bstatus\b", text[m.end():i]), m.group(1)
