"""Registers of the FP64 QR kernels as the compiler reports them. Narrow sketches (several CTAs' shared memory fits
an SM) use kernels of at most 85 registers (128 with panels of 4 or 8 columns), so that three (two) CTAs of 256 threads
share an SM's 65536: with 255 a cooperative QR launch waits until every SM it needs is empty, and a stream of
concurrent requests loses 5 % of its throughput."""
import os
import re
import subprocess

from paper_2606_20195_gb300 import _build


def test_narrow_qr_kernels_leave_room_on_an_sm(tmp_path):
    src = os.path.join(_build.CSRC, "sk_solve.cu")
    r = subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-Xptxas", "-v", "-c", src, "-o",
                        str(tmp_path / "x.o")], capture_output=True, text=True, check=True)
    regs = dict(re.findall(r"Compiling entry function '\w*qr64_kernel(\w+?)EEv.*?Used (\d+) registers",
                           r.stdout + r.stderr, flags=re.S))
    wide = [k for k in regs if k.endswith("Li1E")]
    narrow = [k for k in regs if k not in wide]
    assert len(narrow) == 12 and len(wide) == 4, regs
    assert all(int(regs[k]) <= (85 if "Li16E" in k else 128) for k in narrow), regs
