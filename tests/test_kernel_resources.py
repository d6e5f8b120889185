"""What the compiler reports of the kernels (no GPU): no kernel copies its mesh
descriptor, a parameter, into local memory."""
import os
import re
import subprocess
from concurrent.futures import ThreadPoolExecutor

import kernel_units
from paper_2508_13705_gb300 import build

UNITS = ["inst_1_1_f.cu", "inst_1_1_d.cu", "inst_2_2_f.cu", "inst_2_2_d.cu"]


def stack_frames(unit):
    r = subprocess.run([build._nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-Xptxas", "-v", "-cubin", "-o", os.devnull,
                        os.path.join(build.SRC, unit)], check=True, capture_output=True, text=True)
    return re.findall(r"Function properties for (\w+)\s+(\d+) bytes stack frame", r.stderr)


def test_no_kernel_copies_its_descriptor():
    size = kernel_units.lib().unit_descriptor_bytes()
    with ThreadPoolExecutor(len(UNITS)) as ex:
        for unit, frames in zip(UNITS, ex.map(stack_frames, UNITS)):
            assert len(frames) > 20, unit
            big = {name: int(b) for name, b in frames if int(b) >= size}
            assert not big, (unit, size, big)
