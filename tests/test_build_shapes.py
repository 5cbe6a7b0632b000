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
template <class P, class R, int CS> void lanes(const char* name) {
  using L = mg::HsLayout<P, R, CS>;
  std::printf("%s", name);
  for (int nu = 1; nu <= L::EVCAP; ++nu) std::printf(" %d", mg::hs_lanes<P, L>(nu));
  std::printf("\n");
}
int main() {
  lanes<mg::Proc1, double, mg::CS_SIMT>("lanes_1_fp64");
  lanes<mg::Proc1, float, mg::CS_SIMT>("lanes_1_mixed");
  lanes<mg::Proc2, double, mg::CS_SIMT>("lanes_2_fp64");
  lanes<mg::Proc2, float, mg::CS_SIMT>("lanes_2_mixed");
  lanes<mg::Proc2, float, mg::CS_TC>("lanes_2_tc");
  show<mg::Proc1, float, mg::CS_SIMT, true>("p1_fused");
  show<mg::Proc4, float, mg::CS_SIMT, false>("p4_simt");
  show<mg::Proc4, float, mg::CS_TC, false>("p4_tc");
  show<mg::Proc3, float, mg::CS_SIMT, false>("p3_simt");
  show<mg::Proc3, float, mg::CS_TC, false>("p3_tc");
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


def test_warps_of_small_groups_hold_one_vertex_type(tmp_path):
    """e+e- -> mu+mu- and gg -> t t~ have a dozen items per phase: a group of one
    event would put all of them on one warp, every vertex type after the other."""
    checked = 0
    for name, lanes in layouts(tmp_path).items():
        if not name.startswith("lanes_"):
            continue
        pid = int(name.split("_")[1])
        text = open(os.path.join(B.CSRC, "gen", "proc%d.cuh" % pid)).read()
        table = re.search(r"kHsItems%d\[\d+\] = \{(.*?)\};" % pid, text).group(1)
        types = [int(m.group(1)) for m in re.finditer(r"\{\d+, \{[^}]*\}, (\d+),", table)]
        levels = [int(x) for x in re.search(r"hs_level\(int i\) \{\s*constexpr int t\[\d+\] = \{([^}]*)\}", text).group(1).split(",")]
        for i0, i1 in zip(levels[1:], levels[2:] + [len(types)]):
            for nu, nl in zip(range(1, len(lanes) + 1), lanes):
                assert nl >= nu
                for w in range(0, (i1 - i0) * nl, 32):
                    held = {types[i0 + t // nl] for t in range(w, min(w + 32, (i1 - i0) * nl)) if t % nl < nu}
                    assert len(held) <= (1 if nu <= 8 else 2), (name, nu, nl, held)
                    checked += 1
    assert checked


@pytest.mark.parametrize("name,ctas", [("p4_simt", 1), ("p4_tc", 2), ("p3_simt", 2), ("p3_tc", 3)])
def test_layouts_fit_the_ctas_they_are_built_for(tmp_path, name, ctas):
    """Pairs of events in one CTA of 256 threads per SM for gg -> t t~ g g and two for
    gg -> t t~ g; single events with the tensor-core colour sum in two and three: each
    layout's own count, not that of the process's other kernel."""
    nbytes, _, _, built_for = layouts(tmp_path)[name]
    assert built_for == ctas
    assert (nbytes + CTA_RESERVED) * ctas <= SM_BYTES, nbytes
