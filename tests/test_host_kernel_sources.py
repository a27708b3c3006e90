"""A rule on the device code that no run can show to hold: every kernel may become resident while the one before it in the
stream still writes (programmatic launches), so what another kernel may have written must not be read through the read-only
path, which requires data that nobody writes while the kernel lives, nor with loads that may move above the wait.  The plan's
tables are complete before any launch and may."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_21788_b200", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
# rows of the plan's tables, and the tables themselves
TABLE_ROWS = {"U", "Q", "G"}
TABLES = {"units", "slot_offset", "slot_rows"}
TABLE_ARGS = {"a.work", "a.first_query", "a.row_limit", "a.units", "a.qranges", "a.groups"}


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        s = f.read()
    return re.sub(r"/\*.*?\*/|//[^\n]*", "", s, flags=re.S)


@pytest.mark.parametrize("name", FILES)
def test_read_only_loads_are_for_the_plan_tables(name):
    code = _code(name)
    for arg in re.findall(r"__ldg\(\s*([A-Za-z_][\w.]*)", code):
        assert arg in TABLE_ROWS | TABLES | TABLE_ARGS, arg
    assert len(re.findall(r"__ldg\(", code)) == len(re.findall(r"__ldg\(\s*[A-Za-z_]", code))
    assert not re.findall(r"__ldc[agsv]\s*\(|__ldlu\s*\(|ld\.global\.nc", code)


@pytest.mark.parametrize("name", FILES)
def test_no_kernel_parameter_but_the_plan_tables_is_declared_read_only(name):
    for params in re.findall(r"__global__[^;{]*?\bfcp_\w+\(([^{;]*)\)\s*\{", _code(name), flags=re.S):
        for arg in re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", params):
            assert arg in TABLES, arg


def test_the_rule_sees_the_kernels():
    code = "".join(_code(f) for f in FILES)
    assert len(re.findall(r"__global__[^;{]*?\bfcp_\w+\(([^{;]*)\)\s*\{", code, flags=re.S)) == 6
    assert code.count("__ldg(") > 20


@pytest.mark.parametrize("name", FILES)
def test_the_wait_for_tensor_memory_loads_names_the_registers_they_fill(name):
    """A load from tensor memory fills its registers until the wait behind it, but to the compiler it has written them at once: only
    what passes through the wait is sure to be used behind it."""
    code = _code(name)
    assert not re.findall(r"tc_wait_ld\(\s*\)", code)
    waited = set(re.findall(r"\b(\w+)\)*\s*\)\s*;", " ".join(re.findall(r"tc_wait_ld\([^;]*\);", code))))
    filled = set(re.findall(r"tmem_ld(?:32|16)\([^;]*?(?:, |&)(\w+)(?:\[[^;]*)?\)+;", code)) | set(re.findall(r"\bload\((\w+),", code))
    assert filled <= waited, filled - waited
