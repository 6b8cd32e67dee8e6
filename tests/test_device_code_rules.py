"""Rules that the device code keeps everywhere and that a compiler does not check, read off the sources (no GPU needed)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_05567_b200", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def _code(path):
    """The file without its comments, line structure kept."""
    text = re.sub(r"/\*.*?\*/", lambda m: "\n" * m.group().count("\n"), open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_the_optional_status_word_is_stored_to_in_one_place_only(path):
    stores = re.findall(r"\*\s*(?:\w+\s*[.]\s*)?dev_status\s*=[^=]", _code(path))
    assert len(stores) == (1 if path.endswith("common.cuh") else 0), stores      # common.cuh: report_status, which tests it


def _functions(code):
    """(signature, body) of every __global__ function."""
    for m in re.finditer(r"__global__", code):
        brace = code.index("{", m.start())
        depth, end = 0, brace
        while True:
            depth += {"{": 1, "}": -1}.get(code[end], 0)
            end += 1
            if depth == 0:
                break
        yield code[m.start():brace], code[brace:end]


@pytest.mark.parametrize("path", [p for p in SOURCES if p.endswith(".cu")], ids=os.path.basename)
def test_chained_kernels_read_with_ordinary_loads(path):
    """A kernel that is set up while its predecessor still writes must not use the read-only path (see launch_chained)."""
    chained = [f for f in _functions(_code(path)) if "chain_wait()" in f[1]]
    for signature, body in chained:
        assert not re.search(r"const\s+[\w:]+\s*\*\s*(?:const\s+)?__restrict__", signature + body), signature
        assert "__ldg(" not in body, signature
    helpers = _code(path)
    for _, body in _functions(_code(path)):
        helpers = helpers.replace(body, "")
    assert "__ldg(" not in helpers                  # what kernels call
