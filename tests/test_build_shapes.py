"""Shapes of the helicity-shared kernels against an SM's registers and shared
memory (no GPU needed: nvcc and ptxas only)."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2106_12631_gb300 import build as B

pytestmark = [pytest.mark.slow,
              pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                                 reason="nvcc not available")]

SM_REGISTERS, SM_BYTES, CTA_RESERVED = 65536, 233472, 1024

PROBE = r'''
#include "sigmakin_hs.cuh"
#include "process.cuh"
#include <cstdio>
template <class P, class R, int CS, bool FUSED> void show(const char* name) {
  using L = mg::HsLayout<P, R, CS, FUSED>;
  std::printf("%s %zu %d %d %d\n", name, (size_t)L::bytes, L::NT, L::EVCAP * L::EW, L::H::CTAS);
}
int main() {
  show<mg::Proc1, float, mg::CS_SIMT, true>("p1_fused");
  return 0;
}
'''


def layouts(tmp_path):
    """name -> (bytes of shared memory, threads, events at most, CTAs per SM it is built for)"""
    src, exe = tmp_path / "probe.cu", tmp_path / "probe"
    src.write_text(PROBE)
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    return {ln.split()[0]: tuple(int(x) for x in ln.split()[1:]) for ln in out.split("\n") if ln}


def registers(tmp_path, source, kernel):
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-Xptxas", "-v", "-c", os.path.join(B.CSRC, source), "-o",
                        str(tmp_path / "x.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    m = re.search(r"entry function '\w*%s\w*'.*?Used (\d+) registers" % kernel, r.stderr, re.S)
    return int(m.group(1))


def test_fused_rambo_lanes(tmp_path):
    """RAMBO inside the kernel runs on one lane per event while the CTA's other
    threads wait, so an SM needs many events in flight: at least 128 for
    e+e- -> mu+mu- (4 good helicities of 16; with 64 the call takes half as long
    again)."""
    nbytes, nt, events, _ = layouts(tmp_path)["p1_fused"]
    regs = registers(tmp_path, "sigmakin_p1.cu", "sigmakin_hs_rambo_kernelINS_5Proc1EfLi0E")
    ctas = min(SM_REGISTERS // ((regs + 7) // 8 * 8 * nt), SM_BYTES // (nbytes + CTA_RESERVED))
    assert ctas * min(events, nt // 4) >= 128, (ctas, events, nt, regs)
