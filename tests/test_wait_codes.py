"""Status words of the bounded waits: one value per role and kernel, and only the first role that gives up writes."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_06629_b200", "csrc")


def _read(name):
    return open(os.path.join(CSRC, name)).read()


def test_every_value_belongs_to_one_role_of_one_kernel():
    enum = _read("wait_codes.h").split("enum WaitCode {")[1].split("}")[0]
    values = {n: int(v) for n, v in re.findall(r"(WAIT_\w+) = (\d+)", enum)}
    top = values.pop("WAIT_CODE_MAX")
    assert len(set(values.values())) == len(values) and max(values.values()) == top < 64 and min(values.values()) == 1
    used = {}
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cuh"):
            text = _read(name)
            # no kernel overwrites the word, and every wait that can fail names its role
            assert not re.search(r"atomicExch\((p\.)?status", text), name
            for code in re.findall(r"report_expired\((?:p\.)?status, (\w+),", text):
                used.setdefault(code, set()).add(name)
    assert set(used) == set(values)
    assert all(len(files) == 1 for files in used.values()), used
    assert "atomicCAS(status + STATUS_CODE, 0, code)" in _read("wait_codes.h")


def test_the_header_states_the_range_of_the_values():
    hdr = open(os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include", "layerpipe.h")).read()
    top = int(re.search(r"WAIT_CODE_MAX = (\d+)", _read("wait_codes.h")).group(1))
    assert "(values 1..%d:" % top in hdr
