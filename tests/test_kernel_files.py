"""A kernel alone in its source file costs a module's load, about 0.1 ms, in the first call that launches it:
small ones stay with the kernels that every build runs."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_1812_01448_gb300" / "csrc"


def test_the_host_calls_file_holds_no_kernel():
    src = re.sub(r"//.*", "", (CSRC / "ue_api.cu").read_text())
    assert "__global__" not in src
    assert "<<<" not in src
