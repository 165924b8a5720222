"""Resident blocks per SM that the gated sweeps ask of the register allocator (CPU,
no GPU call): three where that measured faster, two elsewhere."""
import subprocess

import pytest

from paper_2409_10729_gb300 import build as B

# (ndim, direction, mode) -> blocks of 128 threads: mode 0 first, 1 middle, 2 last with the stage update, 3 last of an RHS
CASES = [((3, 0, 0), 2), ((3, 1, 1), 3), ((3, 2, 1), 3), ((3, 2, 3), 3), ((2, 0, 0), 2), ((2, 1, 2), 2), ((2, 1, 3), 2)]


@pytest.fixture(scope="module")
def blocks(tmp_path_factory):
    d = tmp_path_factory.mktemp("gated")
    lines = [f'printf("%d\\n", sweep_min_blocks<FORM_GATED, {m}, {dr}, 2, {nd}>() * sweep_threads({dr}) / 128);'
             for (nd, dr, m), _ in CASES]
    (d / "t.cu").write_text('#include <stdio.h>\n#include "sweep.cuh"\nusing namespace mfc5;\nint main() {\n'
                            + "\n".join(lines) + "\n}\n")
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.COMMON, *B.FAST32, str(d / "t.cu"), "-o", str(d / "t")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([str(d / "t")], capture_output=True, text=True, check=True).stdout.split()
    return [int(x) for x in out]


def test_blocks_per_sm(blocks):
    assert blocks == [b for _, b in CASES]
