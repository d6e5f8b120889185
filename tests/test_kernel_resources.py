"""What the compiler reports of the kernels (no GPU): no kernel copies its mesh
descriptor, a parameter, into local memory; and no FP64 2-D flux spills, whose
resident warps shared memory bounds before the registers do."""
import functools
import os
import re
import subprocess
from concurrent.futures import ThreadPoolExecutor

import kernel_units
from paper_2508_13705_gb300 import build

UNITS = ["inst_1_1_f.cu", "inst_1_1_d.cu", "inst_2_2_f.cu", "inst_2_2_d.cu"]


def report(unit):
    r = subprocess.run([build._nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-Xptxas", "-v", "-cubin", "-o", os.devnull,
                        os.path.join(build.SRC, unit)], check=True, capture_output=True, text=True)
    return re.findall(r"Function properties for (\w+)\s+(\d+) bytes stack frame, (\d+) bytes spill stores", r.stderr)


@functools.lru_cache(maxsize=None)
def reports():
    with ThreadPoolExecutor(len(UNITS)) as ex:
        return dict(zip(UNITS, ex.map(report, UNITS)))


def test_no_kernel_copies_its_descriptor():
    size = kernel_units.lib().unit_descriptor_bytes()
    for unit, kernels in reports().items():
        assert len(kernels) > 20, unit
        big = {name: int(frame) for name, frame, _ in kernels if int(frame) >= size}
        assert not big, (unit, size, big)


def test_fp64_2d_fluxes_do_not_spill():
    fluxes = {name: int(spill) for name, _, spill in reports()["inst_2_2_d.cu"] if "k_flux2" in name}
    assert len(fluxes) >= 12
    assert not any(fluxes.values()), fluxes
