"""Launches of the helicity-shared kernels, on a fake CUDA runtime (no GPU needed).

The launcher is compiled and linked against a runtime whose calls are counted
and whose answers the test chooses.

* An error that an earlier call of the program left in the runtime's last-error
  state is not the launch's: one launch, success, and the earlier error is
  still there for the program to find.
* A launch refused with cudaErrorInvalidValue (its shared-memory attribute is
  gone with a device reset) sets the attribute and is made again, once.
* Any other refusal is returned as it is, and no refusal is left behind in the
  last-error state for the next call to find.
* A batch whose choices of helicities and flows one round of CTAs holds is
  spread so that the CTAs' warps, one per event, take the fewest rounds.
* The kernel-split variant's second kernel spreads a small chunk over the SMs.
"""
import os
import shutil
import subprocess

import pytest

from paper_2106_12631_gb300 import build as B

RUNTIME = r'''
#include <cstddef>
// the runtime's entry points by name: every handle and enumeration is a word here
extern "C" {
struct dim3_ { unsigned x, y, z; };
int launches, attributes, refuse, answer, last, ctas, fit = 1;
int cudaLaunchKernel(const void*, dim3_ g, dim3_, void**, size_t, void*) {
  ++launches;
  ctas = g.x;
  if (refuse == 0) return 0;
  --refuse;
  return last = answer;
}
int __cudaLaunchKernel(void* k, dim3_ g, dim3_ b, void** p, size_t n, void* s) { return cudaLaunchKernel(k, g, b, p, n, s); }
int cudaGetLastError() { const int e = last; last = 0; return e; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaFuncSetAttribute(const void*, int, int) { ++attributes; return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 152; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = fit; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = fit; return 0; }
int __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
int cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
static dim3_ grid, block;
static size_t bytes;
static void* stream;
unsigned __cudaPushCallConfiguration(dim3_ g, dim3_ b, size_t n, void* s) { grid = g; block = b; bytes = n; stream = s; return 0; }
int __cudaPopCallConfiguration(dim3_* g, dim3_* b, size_t* n, void** s) { *g = grid; *b = block; *n = bytes; *s = stream; return 0; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
'''

SRC = r'''
#include "process.cuh"
#include "sigmakin_launch.cuh"
#include <cstdio>
extern "C" int launches, attributes, refuse, answer, last;
static void call(int before, int ans, int times) {
  mg::SigArgs a{};
  a.nevt = 1000;
  mg::Couplings<float> cp{};
  launches = attributes = 0;
  last = before; answer = ans; refuse = times;
  const cudaError_t e = mg::launch_sigmakin_hs_variant<mg::Proc1, float, mg::CS_SIMT>(a, cp, 0, nullptr);
  std::printf("%d %d %d %d\n", (int)e, launches, attributes, last);
}
int main() {
  call(cudaSuccess, cudaSuccess, 0);                  // the first on the device
  call(cudaSuccess, cudaSuccess, 0);
  call(cudaErrorInvalidValue, cudaSuccess, 0);        // an earlier error of the program's own
  call(cudaErrorInvalidDevice, cudaSuccess, 0);
  call(cudaSuccess, cudaErrorInvalidValue, 1);        // refused, then accepted
  call(cudaSuccess, cudaErrorInvalidValue, 2);        // refused again
  call(cudaSuccess, cudaErrorLaunchOutOfResources, 1);
  return 0;
}
'''


SPREAD = r'''
#include "process.cuh"
#include "sigmakin_launch.cuh"
#include <cstdio>
extern "C" int ctas, fit;
int main() {
  fit = 5;
  using H = mg::HsCfg<mg::Proc2, float>;
  mg::Couplings<float> cp{};
  int32_t hel;
  for (int n : {64, 700, 1000, 1301, 2001}) {
    mg::SigArgs a{};
    a.nevt = n;
    a.hel_out = &hel;
    mg::launch_sigmakin_hs_variant<mg::Proc2, float, mg::CS_SIMT>(a, cp, 0, nullptr);
    std::printf("%d %d %d %d\n", n, ctas, H::NT / 32, H::EW);
  }
  return 0;
}
'''


def run(tmp_path, source):
    src, fake, exe = tmp_path / "probe.cu", tmp_path / "runtime.cpp", tmp_path / "probe"
    src.write_text(source)
    fake.write_text(RUNTIME)
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-Xptxas", "-O0", "-cudart", "none", str(src), str(fake),
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")
    return [tuple(int(x) for x in ln.split()) for ln in out if ln.strip()]


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="nvcc not available")
def test_launch_errors(tmp_path):
    rows = run(tmp_path, SRC)
    invalid_value, invalid_device, out_of_resources = 1, 101, 701
    #        status            launches attributes last error left
    assert rows == [(0, 1, 1, 0),
                    (0, 1, 0, 0),
                    (0, 1, 0, invalid_value),
                    (0, 1, 0, invalid_device),
                    (0, 2, 1, 0),
                    (invalid_value, 2, 1, 0),
                    (out_of_resources, 1, 0, 0)]


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="nvcc not available")
def test_choices_take_the_fewest_rounds(tmp_path):
    for n, ctas, warps, per_unit in run(tmp_path, SPREAD):
        units = -(-n // per_unit)
        rounds = lambda g: -(-(-(-units // g)) * per_unit // warps)
        assert ctas <= units
        assert rounds(ctas) == min(rounds(152 * k) for k in range(1, 6)), (n, ctas)


SPLIT = r'''
#include "process.cuh"
#include "sigmakin_split.cuh"
#include <cstdio>
extern "C" int ctas;
int main() {
  using H = mg::HsCfg<mg::Proc3, float>;
  mg::SigArgs a{};
  a.nevt = 1 << 20;
  mg::Couplings<float> cp{};
  for (int n : {1, 3, 64, 257, 1000, 2433, 100003}) {
    mg::SplitLaunch<mg::Proc3, float>::amplitudes(a, cp, 0, n, nullptr, nullptr);
    std::printf("%d %d %d %d\n", n, ctas, H::EVMIN, H::EW);
  }
  return 0;
}
'''


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="nvcc not available")
def test_split_chunks_fill_the_sms(tmp_path):
    for n, ctas, group, per_unit in run(tmp_path, SPLIT):
        units = -(-n // per_unit)
        assert ctas == max(-(-units // group), min(units, 152)), (n, ctas)
