"""Kernels whose blocks wait for one another inside a launch read what other SMs
wrote before the wait.  The language promises that such a load is made, and after
the wait, only where it is volatile and a memory access to the compiler: checked
in the source, since a compiler that happens to keep the order shows nothing."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2212_11024_gb300" / "csrc"


def _code(name):
    text = (CSRC / name).read_text()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def _body(code, head):
    at = code.index("{", code.index(head))
    depth = 0
    for i in range(at, len(code)):
        depth += {"{": 1, "}": -1}.get(code[i], 0)
        if depth == 0:
            return code[at:i + 1]


def test_populations_of_several_steps_are_volatile_loads():
    site, row = _code("step_site.cuh"), _code("step_row.cuh")
    for body in (_body(site, "T load_pop("), _body(row, "float one("), _body(row, "f2 two(")):
        assert "if constexpr (L2)" in body and "load_l2(" in body
        assert not re.search(r"__ld\w+\(", body)


def test_load_past_l1_is_a_volatile_memory_access():
    asm = re.findall(r"asm[^;]*;[^;]*;", _body(_code("aa.cuh"), "T load_l2("))
    assert len(asm) == 3
    for a in asm:
        assert a.startswith("asm volatile(") and a.rstrip().endswith(': "memory");') and "ld.global.cg" in a


def test_last_block_of_a_sum_reads_the_stage_so():
    body = _body(_code("adjoint.cu"), "sum_partials_kernel(")
    after = body[body.index("atomicAdd(ticket"):]
    assert "load_l2(stage" in after and not re.search(r"__ld\w+\(", after)
