"""Which device addresses the state set-up kernel reads in place (CPU).

mfc_set_state and mfc_set_state_prim take a device pointer; the kernel may
dereference it only where it is this device's memory, aligned and long enough.
Everything else has to go through a copy, which the runtime checks.  The choice
is plain C++ (csrc/state_source.h): compiled here and asked case by case.
"""
import os
import re
import subprocess

import pytest

from paper_2409_10729_gb300 import build as B

BASE, SIZE = 0x7f0000000000, 1 << 20

# name: (device memory, its device, range, range bytes, map, map bytes, address, bytes, context's device) -> in place
CASES = {
    "whole allocation": ((1, 0, BASE, SIZE, 0, 0, BASE, SIZE, 0), 1),
    "inside an allocation": ((1, 0, BASE, SIZE, BASE, SIZE, BASE + 512, SIZE - 512, 0), 1),
    "second device's context": ((1, 1, BASE, SIZE, 0, 0, BASE, SIZE, 1), 1),
    "another device's memory": ((1, 1, BASE, SIZE, 0, 0, BASE, SIZE, 0), 0),
    "host or managed memory": ((0, 0, BASE, SIZE, 0, 0, BASE, SIZE, 0), 0),
    "unknown address": ((0, 0, 0, 0, 0, 0, BASE, SIZE, 0), 0),
    "misaligned": ((1, 0, BASE, SIZE, 0, 0, BASE + 4, 512, 0), 0),
    "one double too long": ((1, 0, BASE, SIZE, 0, 0, BASE + 8, SIZE, 0), 0),
    "below the allocation": ((1, 0, BASE, SIZE, 0, 0, BASE - 8, 512, 0), 0),
    "beyond the allocation": ((1, 0, BASE, SIZE, 0, 0, BASE + SIZE + 8, 512, 0), 0),
    "length that wraps": ((1, 0, BASE, SIZE, 0, 0, BASE + 8, 2 ** 64 - 8, 0), 0),
    "reservation mapped in part": ((1, 0, BASE, SIZE, BASE, SIZE // 2, BASE, SIZE, 0), 0),
}


@pytest.fixture(scope="module")
def choice(tmp_path_factory):
    d = tmp_path_factory.mktemp("source")
    rows = ",\n".join("{{%s, %d, %dULL, %dULL, %dULL, %dULL}, %dULL, %dULL, %d}" % (("true" if a[0] else "false",) + a[1:])
                      for a, _ in CASES.values())
    (d / "t.cpp").write_text(
        '#include <stdio.h>\n#include "state_source.h"\nusing namespace mfc5;\n'
        "struct Row { PointerInfo p; uintptr_t addr; size_t bytes; int device; };\n"
        f"static const Row rows[] = {{\n{rows}}};\n"
        'int main() { for (const Row& r : rows) printf("%d\\n", (int)read_in_place(r.p, r.addr, r.bytes, r.device)); }\n')
    subprocess.run(["g++", "-std=c++17", "-I", B.CSRC, str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    out = subprocess.run([str(d / "t")], capture_output=True, text=True, check=True).stdout.split()
    return dict(zip(CASES, map(int, out)))


@pytest.mark.parametrize("name", CASES)
def test_read_in_place(choice, name):
    assert choice[name] == CASES[name][1]


def test_state_setters_ask_before_the_kernel_reads_the_callers_address():
    """Both setters go through one function, whose device branch launches on the
    caller's address only where the choice above allows it."""
    src = open(os.path.join(B.CSRC, "capi.cu")).read()
    body = re.search(r"static int set_state_impl\(.*?\n}", src, re.S).group(0)
    guard = body.index("read_in_place(pointer_info(src)")
    copy = body.index("cudaMemcpyAsync(ctx->qn, src")
    assert guard < copy < body.index("set_state_from(ctx, src")
    for name in ("mfc_set_state", "mfc_set_state_prim"):
        assert re.search(r'extern "C" int %s\([^)]*\) \{\s*return set_state_impl\(' % name, src)
