"""Choice between the mixed form's two kernels of a sweep (CPU, no GPU call).

The lean kernel reconstructs one field at a time, along x at two blocks per SM;
the full one packs pairs of fields and may run three.  Which of them a launch
takes is a host rule (lean_use, take_lean); the register allocator says where
packing would spill.
"""
import os
import re
import subprocess

import pytest

from paper_2409_10729_gb300 import build as B


def _nvcc(src, out, *flags):
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.COMMON, *B.FAST32, *flags, str(src), "-o", str(out)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stderr


def test_four_fluid_x_sweeps_do_not_spill(tmp_path):
    src = tmp_path / "x4.cu"
    src.write_text('#include "sweep.cuh"\nnamespace mfc5 {\n'
                   "template cudaError_t launch_kernel<2, 0, SW_FIRST, FORM_MIXED, false, 4>(const SweepArgs&, cudaStream_t);\n"
                   "template cudaError_t launch_kernel<3, 0, SW_FIRST, FORM_MIXED, false, 4>(const SweepArgs&, cudaStream_t);\n}\n")
    info = _nvcc(src, tmp_path / "x4.o", "-Xptxas=-v", "-c")
    stores = [int(x) for x in re.findall(r"(\d+) bytes spill stores", info)]
    assert len(stores) == 2 and not any(stores), info


# (ndim, direction, non-uniform, fluids, order, lean blocks, full blocks, lean taken), for 152 SMs: x blocks are one
# warp, 8 resident per SM at two blocks of 128 and 12 at three; y blocks 16 warps per SM (z and the 2-D y sweep 12)
RULE = [
    (2, 0, False, 2, 3, 32, 32, 1),          # 64x48
    (2, 0, False, 2, 3, 1216, 1216, 1),      # the last size that both hold in one wave
    (2, 0, False, 2, 3, 1600, 1600, 0),      # 640x320: two waves against one
    (2, 0, False, 2, 3, 2048, 2048, 1),      # 2048x1024: two waves both ways
    (2, 0, False, 2, 5, 32, 32, 0),          # WENO5 never
    (3, 0, False, 2, 3, 256, 256, 1),        # 32^3
    (3, 0, False, 2, 3, 608, 608, 1),        # half a wave (3-D x: two blocks either way)
    (3, 0, False, 2, 3, 609, 609, 0),
    (3, 0, False, 2, 3, 2048, 2048, 0),      # 64^3
    (3, 1, False, 2, 3, 304, 304, 1),
    (3, 1, False, 2, 3, 305, 305, 0),
    (3, 0, True, 2, 5, 2048, 2048, 1),       # 128^3: two waves both ways
    (3, 0, True, 2, 5, 1728, 1728, 0),       # 96^3: two against one
    (2, 0, False, 3, 3, 1600, 1600, 1),      # three fluids in 2-D: WENO3 lean, WENO5 full
    (2, 0, False, 3, 5, 1600, 1600, 0),
]
USE = [((2, 0, 0, 4), 1), ((3, 0, 0, 4), 1), ((3, 1, 0, 4), 0), ((3, 0, 0, 3), 0), ((2, 0, 0, 3), 2), ((2, 1, 0, 3), 0),
       ((3, 2, 0, 2), 2), ((1, 0, 0, 2), 0), ((3, 0, 1, 2), 2), ((3, 1, 1, 2), 0)]


@pytest.fixture(scope="module")
def answers(tmp_path_factory):
    d = tmp_path_factory.mktemp("lean")
    lines = []
    for nd, dr, nu, nf, order, lb, fb, _ in RULE:
        ls = 152 * (8 if dr == 0 else 4)
        fs = 152 * (12 if dr == 0 and (nu or nd == 2) else 8 if dr == 0 else 4)
        lines.append(f'printf("%d\\n", (int)take_lean({nd}, {dr}, {int(nu)}, {nf}, {order}, {{{lb}, {ls}}}, {{{fb}, {fs}}}));')
    for (nd, dr, nu, nf), _ in USE:
        lines.append(f'printf("%d\\n", (int)lean_use(FORM_MIXED, {nd}, {dr}, {nu}, {nf}));')
        lines.append(f'printf("%d\\n", (int)lean_use(FORM_GATED, {nd}, {dr}, {nu}, {nf}));')
    (d / "t.cu").write_text('#include <stdio.h>\n#include "mfc_internal.cuh"\nusing namespace mfc5;\nint main() {\n'
                            + "\n".join(lines) + "\n}\n")
    _nvcc(d / "t.cu", d / "t")
    return [int(x) for x in subprocess.run([str(d / "t")], capture_output=True, text=True, check=True).stdout.split()]


def test_launches_take_the_kernel_that_measured_faster(answers):
    assert answers[:len(RULE)] == [r[-1] for r in RULE]


def test_variants_exist_only_where_there_is_a_choice(answers):
    got = answers[len(RULE):]
    assert got[0::2] == [u for _, u in USE]
    assert not any(got[1::2])   # the gated form has none
