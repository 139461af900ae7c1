"""What the sources promise about data that an earlier kernel of the stream may still be writing when a kernel starts (no GPU:
a race cannot be shown by running it)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_30386_b200", "csrc")
# device tables of a plan and names for parts of them: written before the first launch that can name them, never after
PLAN_TABLES = {"row_src", "row_pos", "layer_row_off", "src_l", "pos_l"}


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _launched_in_order():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu") and "launch_in_order(" in _code(f))


def test_every_kernel_source_is_looked_at():
    assert _launched_in_order() == ["codec_int8.cu", "pack_restore.cu", "refresh_chunked.cu", "refresh_seq.cu"]


@pytest.mark.parametrize("name", _launched_in_order())
def test_only_plan_tables_take_the_non_coherent_path(name):
    code = _code(name)
    assert not re.search(r"ld\.global\.nc|ld\.global[.\w:]*\.nc\b", code)
    for arg in re.findall(r"__ldg\(([^;]*)", code):
        first = re.match(r"(?:reinterpret_cast<[^>]*>\()?(\w+)", arg).group(1)
        assert first in PLAN_TABLES, f"__ldg({arg[:40]}"
    for param in re.findall(r"__restrict__\s+(\w+)", code):
        assert param in PLAN_TABLES, param


def test_plan_tables_are_on_the_device_when_the_plan_is_returned():
    body = re.search(r"dasc_status_t attach_device\(.*?\n}\n", _code("dasc_api.cu"), flags=re.S).group(0)
    last_copy = max(m.start() for m in re.finditer(r"upload\(", body))
    assert re.search(r"cuda(Stream|Device)Synchronize\(", body[last_copy:])
