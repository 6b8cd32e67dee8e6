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
