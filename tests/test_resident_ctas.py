"""compress_fused is launched with as many CTAs as fit the SMs.  How many do follows from the kernel's static shared memory and registers,
which the compiler reports, and from the dynamic shared memory of the launch; here against the launch's own estimate."""
import os
import re
import subprocess

from paper_2605_22718_b200.build import CSRC, NVCC_FLAGS, ROOT, _nvcc

SM_BYTES, RESERVED = 228 * 1024, 1024      # shared memory of an SM; what the system keeps of it per CTA
SM_REGISTERS, THREADS = 65536, 256


def test_ctas_that_the_one_launch_kernel_plans_for(tmp_path):
    flags = [f for f in NVCC_FLAGS if f not in ("-shared", "-lineinfo")]
    source = os.path.join(CSRC, "wk_compress.cu")
    out = subprocess.run([_nvcc(), *flags, "-cubin", "-I", os.path.join(ROOT, "include"), "-o", str(tmp_path / "k"), source], check=True,
                         stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True).stdout
    entry = r"entry function '\S*compress_fused\S*' for(?:(?!entry function).)*?Used (\d+) registers[^\n]*?(\d+) bytes smem"
    kernels = [(int(r), int(s)) for r, s in re.findall(entry, out, re.S)]
    assert len(kernels) == 4
    sm, static_kb = re.search(r"kSmBytes = (\d+) \* 1024, kFusedStatic = (\d+) \* 1024", open(source).read()).groups()
    for regs, static in kernels:
        by_registers = SM_REGISTERS // (THREADS * ((regs + 7) // 8 * 8))
        for dynamic in range(16 * 1024, 220 * 1024, 256):
            planned = min(int(sm) * 1024 // (dynamic + int(static_kb) * 1024), by_registers)
            assert SM_BYTES // (static + dynamic + RESERVED) >= planned, (static, dynamic)
