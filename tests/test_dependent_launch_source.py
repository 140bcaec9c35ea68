"""What a kernel launched as a programmatic dependent launch may promise the compiler.

Such a kernel is resident while the launch before it still writes the state.  A `__restrict__` pointer
or an `__ldg` promises data that no one writes for the kernel's whole lifetime, which lets the loads move
above the wait and through a cache that need not see the writes.  Only what no launch writes (node
flags, the wall list) may be read so.  The failure would be a race on memory, so it is looked for in
the source, not provoked."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_22256_gb300", "csrc")
STATIC = {"flags", "a.wsub", "wax", "way"}  # written at creation only


def waiting_kernels():
    """(file, name, parameters, body) of every kernel that calls pdl_wait()."""
    found = []
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for part in re.split(r"(?=__global__)", text)[1:]:
            m = re.match(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)\s*)?(\w+)\(([^)]*)\)\s*\{", part)
            if not m:
                continue
            body = part[m.end():part.index("\n}", m.end())]
            if "pdl_wait()" in body:
                found.append((name, m.group(1), m.group(2), body))
    return found


def test_the_kernels_are_found():
    assert {k[1] for k in waiting_kernels()} == {"k_step", "k3_rho", "k3_march"}


@pytest.mark.parametrize("kernel", waiting_kernels(), ids=lambda k: k[1])
def test_only_data_that_no_launch_writes_is_promised_constant(kernel):
    _, name, params, body = kernel
    promised = {p.split()[-1] for p in params.split(",") if "__restrict__" in p}
    assert promised <= STATIC, (name, promised - STATIC)
    read_only = {m.strip() for m in re.findall(r"__ldg\(\s*([\w.]+)", body)}
    assert read_only <= STATIC, (name, read_only - STATIC)
