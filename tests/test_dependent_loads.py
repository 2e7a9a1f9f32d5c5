"""Source rule of dependent launches (csrc/launch.cuh): a kernel that may start while its
predecessor runs reads and writes tensor data through plain pointers. The compiler may
move a load through a __restrict__ pointer, or through the read-only path, above the wait
for the predecessor; only tables that the host uploaded may be read that way."""

import os
import re

import paper_2205_00393_gb300

CSRC = os.path.join(os.path.dirname(paper_2205_00393_gb300.__file__), "csrc")
TABLES = {"GemmParams", "int2", "int", "int64_t", "RootParams", "PermParams", "StemParams", "StemRegBranches",
          "LeafEnvParams", "InvEnvParams", "double2* const"}  # (the last: a table of pointers)


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_dependent_kernels_read_data_through_plain_pointers():
    files = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
    text = {f: _source(f) for f in files}
    dependent = set(re.findall(r"launch_dependent\(\s*(k_\w+)", "\n".join(text.values())))
    assert len(dependent) > 15
    seen = set()
    for f in files:
        src = text[f]
        assert not re.search(r"__ldg|\.nc\.", src), f
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\(([^{;]*?)\)\s*[{;]", src, re.S):
            if m.group(1) not in dependent:
                continue
            seen.add(m.group(1))
            for arg in m.group(2).split(","):
                if "__restrict__" in arg:
                    kind = re.sub(r"\s*\*\s*__restrict__.*", "", arg.strip().removeprefix("const ")).strip()
                    assert kind in TABLES, (f, m.group(1), arg.strip())
        # device code outside kernel signatures: tables only
        body = re.sub(r"__global__[^;{]*?\bk_\w+\([^{;]*?\)\s*[{;]", "", src, flags=re.S)
        for m in re.finditer(r"(\w+)\s*\*\s*__restrict__", body):
            assert m.group(1) in TABLES, (f, m.group(0))
    assert seen == dependent
