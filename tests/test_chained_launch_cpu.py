"""The rule behind launches that may start before their predecessor ends, checked on the source: the launch attribute is set
in one place, from a flag of the caller (the ragged batch's parallel branches turn it off), and every kernel launched so
waits for its predecessor in its first statement, through every pointer that it is given, before it lets its successor
start."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2210_09196_gb300" / "csrc"
SOURCES = {p.name: re.sub(r"//[^\n]*", "", p.read_text()) for p in sorted([*CSRC.glob("*.cu"), *CSRC.glob("*.cuh")])}


def test_the_attribute_is_set_in_one_place_from_the_callers_flag():
    named = [n for n, s in SOURCES.items() if "ProgrammaticStreamSerialization" in s]
    assert named == ["internal.cuh"]
    assert re.findall(r"programmaticStreamSerializationAllowed = ([^;]+);", SOURCES["internal.cuh"]) == ["chained ? 1 : 0"]


def kernels():
    out = []
    for n, s in SOURCES.items():
        for m in re.finditer(r"__global__", s):
            body = s.index("{", m.end())
            name, args = re.search(r"(\w+_kernel)\s*\((.*)\)\s*$", s[m.end():body], re.S).groups()
            out.append((n, name, args, s[body + 1:body + 600]))
    return out


PLAIN = {"tune_fill_kernel", "dmrs_type1_kernel", "noalloc_twiddle_kernel", "noalloc_status_kernel", "selftest_wait_kernel"}


def test_the_other_kernels_are_launched_in_order():
    launched = {m for s in SOURCES.values() for m in re.findall(r"(\w+_kernel)(?:<[^;{}]*?>)?<<<", s)}
    assert launched == PLAIN


@pytest.mark.parametrize("where,name,args,body", [k for k in kernels() if k[1] not in PLAIN], ids=lambda v: v if str(v).endswith("_kernel") else "")
def test_a_chained_kernel_waits_first(where, name, args, body):
    m = re.match(r"\s*(?:pusch::)?chain_wait\(([^)]*)\);", body)
    assert m, (where, name)
    pointers = {p.split("*")[-1].replace("__restrict__", "").strip() for p in args.split(",") if "*" in p}
    assert pointers == {v.strip() for v in m.group(1).split(",")}
    go = body.find("chain_go()")
    assert go < 0 or go > m.end() - 1
