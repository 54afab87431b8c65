"""Rules of the device code that no run can show, checked on its text.

No tensor or bulk copy goes to several CTAs at once: the library also runs with
one rank per GPU (`bench.py` under torchrun), where such copies are not used.

Explicit read-only loads (ld.global.nc, __ldg) are for weights alone: with
programmatic dependent launch a kernel starts while the one before still writes
its activations, and PTX allows such loads only of memory that nobody writes while
the kernel runs.
"""

import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2508_06024_gb300" / "csrc"
FILES = sorted(p for p in CSRC.iterdir() if p.suffix in (".cu", ".cuh"))


def _code(path):
    """The file without comments, adjacent string literals joined."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", path.read_text(), flags=re.S)
    return re.sub(r'"\s*"', "", text)


@pytest.mark.parametrize("path", FILES, ids=lambda p: p.name)
def test_copies_have_one_destination(path):
    for copy in re.findall(r"cp\.async\.bulk[^;]*;", _code(path)):
        assert "multicast" not in copy, copy


@pytest.mark.parametrize("path", FILES, ids=lambda p: p.name)
def test_read_only_loads_are_of_weights(path):
    code = _code(path)
    assert not re.findall(r"\bld\.global[.\w]*\.nc\b", code)
    lines = [line for line in code.splitlines() if "__ldg(" in line]
    # the weight rows of the fp32 GEMM
    assert all("rb[i]" in line for line in lines), lines
