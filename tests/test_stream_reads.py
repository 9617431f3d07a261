"""Kernels launched to overlap the work before them may be resident while that work still
writes what they read, so they must not read it through the read-only data path.  The sources
use that path only in two diagnostics, and by ld_input<kReadOnly> in the kernels that are
launched the ordinary way."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1202_6163_gb300", "csrc")
DIAGNOSTICS = ("k_probe_l2", "k_tile_weights")
READ_ONLY = re.compile(r"__ldg\s*\(|ld\.global\.nc|__restrict__")


def code(path):
    """The file without its comments."""
    text = open(path).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", lambda m: "\n" * m.group(0).count("\n"), text, flags=re.S)


def body(text, at):
    """Start and end of the definition whose head matches at `at`."""
    i = text.index("{", at.end())
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
    return at.start(), j


def head(text, name, kind="__global__"):
    return re.search(kind + r"[^;{}]*\b" + name + r"\s*\(", text)


def sources():
    return {os.path.basename(p): code(p)
            for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))}


def overlapped():
    text = "\n".join(sources().values())
    names = set(re.findall(r"\b(k_\w+)\b", " ".join(re.findall(r"launch_overlapped\(([^;]*);", text))))
    assert len(names) >= 12, names
    return text, names | {"k_small"}  # launched with the attribute by itself


def test_read_only_path_only_behind_ld_input():
    found = []
    for file, text in sources().items():
        for name, kind in [(n, "__global__") for n in DIAGNOSTICS] + [("ld_input", "__device__")]:
            at = head(text, name, kind)
            if at:
                i, j = body(text, at)
                text = text[:i] + text[j:]
        found += [(file, m.group(0)) for m in READ_ONLY.finditer(text)]
    assert not found


def test_overlapped_kernels_wait_first_and_read_the_ordinary_way():
    text, names = overlapped()
    assert not names & set(DIAGNOSTICS)
    for name in names:
        at = head(text, name)
        assert at, name
        i, j = body(text, at)
        assert "grid_begin();" in text[i:j], name
        assert "kReadOnly" not in text[i:j] and not re.search(r"(ld_input|read_logw)<true>", text[i:j]), name

