"""Registers that nvcc reports for kernels whose speed hangs on the number of
CTAs that an SM holds (65,536 registers)."""
import functools
import os
import re
import subprocess

from paper_2509_15744_gb300 import build


@functools.lru_cache
def _log(source):
    cmd = [build._nvcc(), *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c", os.path.join(build.CSRC, source), "-o",
           os.devnull]
    return subprocess.run(cmd, capture_output=True, text=True, check=True).stderr


def _resources(source, kernel):
    """{(order, type, further template argument): (registers, spill bytes)} of a velocity kernel."""
    out = {}
    for name, spill, regs in re.findall(
            r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores.*?Used (\d+) registers", _log(source),
            flags=re.S):
        m = re.search(kernel + r"_kernelILi(\d)E(6__half|13__nv_bfloat16)Li(\d+)E(?:Li(\d)E)?", name)
        if m:
            out[2 * int(m[1]), m[2].lstrip("0123456789"), m[4]] = (int(regs), int(spill))
    return out


def test_16_bit_3d_steps_hold_the_ctas_that_hide_their_latency():
    res = _resources("step_velocity.cu", "step3d_velocity")
    for t in ("__half", "__nv_bfloat16"):
        of = {o: [v for (order, typ, _), v in res.items() if (order, typ) == (o, t)] for o in (2, 4, 6, 8)}
        # orders 2 and 4: four CTAs of 256 threads without being held to it
        for o in (2, 4):
            assert [v for v in of[o] if v[0] <= 64 and v[1] == 0], (t, o, of[o])
        # orders 6 and 8: four CTAs for grids that fill them, a variant without spills for the others
        for o in (6, 8):
            assert min(v[0] for v in of[o]) <= 64 and [v for v in of[o] if v[1] == 0], (t, o, of[o])


def test_16_bit_2d_steps_hold_the_ctas_that_their_split_counts_on():
    res = _resources("step_velocity.cu", "step2d_velocity")
    for t in ("__half", "__nv_bfloat16"):
        for order, ctas in ((2, 7), (4, 7), (6, 6), (8, 5)):   # of 128 threads, in steps of 8 registers
            (regs, spill), = [v for (o, typ, _), v in res.items() if (o, typ) == (order, t)]
            assert -(-regs // 8) * 8 * 128 * ctas <= 65536 and spill == 0, (t, order, regs, spill)
